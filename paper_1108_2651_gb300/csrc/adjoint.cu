// Reverse-time adjoint of the stream-collide step (not in the paper): the
// gradient of a function of the receiver traces with respect to the relative
// permittivity, for FP32 storage and uniform mu.
//
// Forward map of one step (Eqs. 17-18), site by site: the post-collision
// p^t(y) = M(y) g^t(y) + T^t(y) streams to g^{t+1}_i(y + c_i) = p^t_i(y).
// With lambda^t = dL/dg^t (pre-collision) and mu^t = dL/dp^t:
//   mu^t_i(y)   = lambda^{t+1}_i(y + c_i)                  (transpose of streaming)
//   lambda^t(y) = M(y)^T mu^t(y) + d l_t / d g^t(y)        (receivers at time t)
//   dL/dc_L^2(y) += mu^t(y) . [dM/dc_L^2 g^t(y) + dT^t/dc_L^2(y)] + d l_t/dc_L^2(y)
// M = 2P - I with P the equilibrium map of Eq. 8.  Written out (tau = dt/2,
// moving weights c_L^2/2, w0 = 1 - D c_L^2, nu = sum_i w_i mu_i):
//   2D:  lambda_0 = 2 nu - mu_0,  lambda_1 = 2 nu - mu_3,  lambda_3 = 2 nu - mu_1,
//        lambda_2 = 2 nu - mu_4,  lambda_4 = 2 nu - mu_2
//   3D:  lambda_{0a} = 2 nu_a - mu_{0a},
//        lambda_{ja} = 2 nu_a + (c_j x V)_a / 2 - mu_{ja},  V = sum_i mu_i x c_i
// and, with sigma = sum_i g_i (per component) and j the point current,
//   2D:  dM g/dc_L^2 = sigma (moving), -4 sigma (rest);  dT/dc_L^2 = j/2, -2 j
//   3D:  dM g/dc_L^2 = sigma (moving), -6 sigma (rest);  dT/dc_L^2 = j/4, -3 j/2
// Receivers: E = -c_L^2 sigma gives d/dg_i = -c_L^2 and d/dc_L^2 = -sigma;
// B components are differences of populations (2D: B_x = g_4 - g_2,
// B_y = g_1 - g_3; 3D: B = sum_i g_i x c_i).  Finally
//   dL/d eps_r = dL/dc_L^2 * dc_L^2/d eps_r = -dL/dc_L^2 * c_L^2 / eps_r.
//
// Of a state g^t the adjoint needs sigma only: 3 words a site in 3D against the
// state's 21.  In 3D the forward kernels write it as they step (the sums are
// those of the collision), and lambda is stored by opposite directions, so that
// its transposed streaming is the forward step's pull and the kernel of several
// steps per launch (march3d.cu) serves both.  lbem_forward_record keeps every
// step's sigma where that takes no more memory than states every K steps and a
// segment of K states would (3 nsteps <= 21 (nsteps / K + K)); the backward pass
// is then one sweep.  Else, and in 2D (a state is 5 words, sigma 1), it
// keeps the state every K steps, and the backward pass recomputes one segment
// of at most K steps at a time: its sigmas in 3D, its states in 2D.  40 steps of
// 96^3 with K = 10 recorded and gone back: 5.23 ms with states kept and
// recomputed, buffers allocated each time and single steps; 2.7 ms with sigmas
// and the last run's buffers; 2.3 ms with three steps per launch (18.5 us a step
// forward, of L2 bandwidth as the steps themselves).  The gradient is accumulated over time steps in FP64; each step's contribution at
// a site is formed in FP32, like the rest of the arithmetic (GB300's FP64 rate
// is a small fraction of its FP32 rate, and the per-site FP64 products had made
// the adjoint step compute-bound).
#include <math.h>

#include <algorithm>
#include <vector>

#include "site3d.cuh"

namespace lbk {

// A run's buffers; the next run of the handle takes them over as far as they are large enough.
struct AdjointState {
    int nsteps = 0, every = 0, ncp = 0;
    long long t0 = 0;
    size_t state_floats = 0, sig_floats = 0;
    bool all = false;       // 3D: seg holds every step's sigma, and there are no checkpoints
    float *cps = nullptr;   // [ncp][state]
    float *seg = nullptr;   // 2D: [every][state]; 3D: sigma of every step, or of a segment's: [..][3][plane]
    float *work = nullptr;  // 3D with checkpoints: [2][state], the states recomputed
    float *lam = nullptr;   // [2][state]
    double *gcl = nullptr;  // [plane]
    float *cot = nullptr;   // [nrec][nsteps]
    float *gout = nullptr;  // [nsite] staging for host outputs
    double *gcl_out = nullptr;
    size_t cps_cap = 0, seg_cap = 0, work_cap = 0, lam_cap = 0, gcl_cap = 0, cot_cap = 0;  // elements
};

// Makes p hold at least need elements (its contents are lost when it has to grow).
template <class T>
static bool ensure(T *&p, size_t &cap, size_t need) {
    if (cap >= need) return true;
    cudaFree(p);
    p = nullptr;
    cap = 0;
    if (cudaMalloc((void **)&p, need * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        p = nullptr;
        return false;
    }
    cap = need;
    return true;
}

void adjoint_free(lbem_t *h) {
    if (!h || !h->adj) return;
    AdjointState *a = h->adj;
    cudaFree(a->cps);
    cudaFree(a->seg);
    cudaFree(a->work);
    cudaFree(a->lam);
    cudaFree(a->gcl);
    cudaFree(a->cot);
    cudaFree(a->gout);
    cudaFree(a->gcl_out);
    delete a;
    h->adj = nullptr;
}

struct AdjArgs {
    Grid g;
    const float *lam_in;  // lambda^{t+1}, site layout [npop][plane]
    float *lam_out;       // lambda^t
    PopBuf state;         // forward buffer at time t (g^t = pull)
    const float *cL2;
    double *gcl;
    Events evt;           // sources (j) and receivers (cotangent)
    const float *cot;     // [nrec][nsteps]
    int nsteps;
    long long t, t0;
};

__device__ __forceinline__ float4 f4(const float *base, long long plane, int p, int row, int pitch, int c) {
    return __ldg(reinterpret_cast<const float4 *>(base + p * plane + (long long)row * pitch) + c);
}
__device__ __forceinline__ float f1(const float *base, long long plane, int p, int row, int pitch, int x) {
    return __ldg(base + p * plane + (long long)row * pitch + x);
}

// Element x of plane p shifted by one site: want = +1 gives v(x+1), -1 gives v(x-1),
// for the 4 sites of this lane (all 32 lanes must call).
__device__ __forceinline__ float4 xshift(const float *base, long long plane, int p, int row, const Grid &G, int c,
                                         int lane, int want, bool active) {
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 a = active ? f4(base, plane, p, row, G.pitch, c) : z4;
    const int x0 = 4 * c;
    if (want < 0) {
        float prev = __shfl_up_sync(FULL, a.w, 1);
        if (lane == 0 && active) prev = f1(base, plane, p, row, G.pitch, c == 0 ? G.nx - 1 : x0 - 1);
        return make_float4(prev, a.x, a.y, a.z);
    }
    float next = __shfl_down_sync(FULL, a.x, 1);
    if (lane == 31 && x0 + 4 < G.nx) next = f1(base, plane, p, row, G.pitch, x0 + 4);
    float4 r = make_float4(a.y, a.z, a.w, next);
    if (c == G.nchunk - 1) set(r, G.nx - 1 - x0, f1(base, plane, p, row, G.pitch, 0));
    return r;
}

// ------------------------------------------------------------------ 2D
__global__ void __launch_bounds__(BLOCK) adjoint2d(AdjArgs a) {
    const Grid &G = a.g;
    const int lane = threadIdx.x & 31;
    const long long wg = ((long long)blockIdx.x * BLOCK + threadIdx.x) >> 5;
    const int wpr = G.nchunk_pad >> 5;
    const int row = (int)(wg / wpr);
    const int c = (int)(wg - (long long)row * wpr) * 32 + lane;
    if (row >= G.ny) return;
    const bool active = c < G.nchunk;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const int ym = row == 0 ? G.ny - 1 : row - 1, yp = row == G.ny - 1 ? 0 : row + 1;
    const float *L = a.lam_in;
    // mu_i(y) = lambda_i(y + c_i)
    float4 m[5];
    m[0] = active ? f4(L, G.plane, 0, row, G.pitch, c) : z4;
    m[1] = xshift(L, G.plane, 1, row, G, c, lane, +1, active);
    m[2] = active ? f4(L, G.plane, 2, yp, G.pitch, c) : z4;
    m[3] = xshift(L, G.plane, 3, row, G, c, lane, -1, active);
    m[4] = active ? f4(L, G.plane, 4, ym, G.pitch, c) : z4;
    // sigma of g^t(y): g_i(y) = P_i(y - c_i)
    const float *S = static_cast<const float *>(a.state.data);
    float4 sg = active ? f4(S, G.plane, 0, row, G.pitch, c) : z4;
    {
        const float4 s1 = xshift(S, G.plane, 1, row, G, c, lane, -1, active);
        const float4 s3 = xshift(S, G.plane, 3, row, G, c, lane, +1, active);
        const float4 s2 = active ? f4(S, G.plane, 2, ym, G.pitch, c) : z4;
        const float4 s4 = active ? f4(S, G.plane, 4, yp, G.pitch, c) : z4;
        sg = make_float4(((sg.x + s1.x) + (s2.x + s3.x)) + s4.x, ((sg.y + s1.y) + (s2.y + s3.y)) + s4.y,
                         ((sg.z + s1.z) + (s2.z + s3.z)) + s4.z, ((sg.w + s1.w) + (s2.w + s3.w)) + s4.w);
    }
    if (!active) return;
    const float4 cl = f4(a.cL2, 0, 0, row, G.pitch, c);
    float4 jz = z4;
    float4 o[5];
    float dg[4] = {0.f, 0.f, 0.f, 0.f};  // this step's contribution, FP32; accumulated over steps in FP64
    for (int j = 0; j < 4; j++) {
        const float q = get(cl, j), w0 = 1.f - 2.f * q;
        const float mm = ((get(m[1], j) + get(m[2], j)) + get(m[3], j)) + get(m[4], j);
        const float nu = w0 * get(m[0], j) + 0.5f * q * mm;
        set(o[0], j, 2.f * nu - get(m[0], j));
        set(o[1], j, 2.f * nu - get(m[3], j));
        set(o[3], j, 2.f * nu - get(m[1], j));
        set(o[2], j, 2.f * nu - get(m[4], j));
        set(o[4], j, 2.f * nu - get(m[2], j));
        const float s = get(sg, j);
        dg[j] = s * mm - 4.f * (s * get(m[0], j));
    }
    if (a.evt.rowptr) {
        const int e0 = __ldg(a.evt.rowptr + row), e1 = __ldg(a.evt.rowptr + row + 1);
        for (int e = e0; e < e1; e++) {
            const Event ev = a.evt.ev[e];
            if ((ev.x >> 2) != c) continue;
            const int j = ev.x & 3;
            if (ev.kind == 0) {
                if (ev.comp == 2 && a.t < a.evt.nt) set(jz, j, get(jz, j) + __ldg(a.evt.amp + (long long)ev.index * a.evt.nt + a.t));
            } else {
                const long long n = a.t - a.t0;
                if (n < 0 || n >= a.nsteps || a.t >= a.evt.cap) continue;
                const float r = __ldg(a.cot + (long long)ev.index * a.nsteps + n);
                if (ev.comp == 2) {  // E_z = -c_L^2 sigma
                    const float d = -get(cl, j) * r;
                    for (int i = 0; i < 5; i++) set(o[i], j, get(o[i], j) + d);
                    dg[j] -= get(sg, j) * r;
                } else if (ev.comp == 3) {  // B_x = g_4 - g_2
                    set(o[4], j, get(o[4], j) + r);
                    set(o[2], j, get(o[2], j) - r);
                } else if (ev.comp == 4) {  // B_y = g_1 - g_3
                    set(o[1], j, get(o[1], j) + r);
                    set(o[3], j, get(o[3], j) - r);
                }
            }
        }
    }
    for (int j = 0; j < 4; j++) {
        const float mm = ((get(m[1], j) + get(m[2], j)) + get(m[3], j)) + get(m[4], j);
        dg[j] += get(jz, j) * (0.5f * mm - 2.f * get(m[0], j));
        const int x = 4 * c + j;
        if (x < G.nx) a.gcl[(long long)row * G.pitch + x] += (double)dg[j];
    }
    for (int i = 0; i < 5; i++) Codec<LBEM_F32>::store4(PopBuf{a.lam_out, nullptr, G.plane, 0, G.pitch, 0}, i, row, c, o[i]);
}

// ------------------------------------------------------------------ 3D
// One site per thread; the same update as the kernel of several steps per launch.  lambda is stored by opposite
// directions, so mu is pulled as the forward step pulls.  The FP64 gradient accumulator is loaded with the other operands,
// at the top, so its latency overlaps theirs.  MINB = 5 caps the registers (handle variant 2).
template <int MINB>
__global__ void __launch_bounds__(BLOCK, MINB) adjoint3d_site(AdjArgs a, const float *sig) {
    const Grid &G = a.g;
    int row, x;
    site_of(G, row, x);
    if (row >= G.nrows || x >= G.nx) return;
    const int z = row / G.ny, y = row - z * G.ny;
    const int rym = z * G.ny + (y == 0 ? G.ny - 1 : y - 1), ryp = z * G.ny + (y == G.ny - 1 ? 0 : y + 1);
    const int rzm = (z == 0 ? G.nz - 1 : z - 1) * G.ny + y, rzp = (z == G.nz - 1 ? 0 : z + 1) * G.ny + y;
    const int xm = x == 0 ? G.nx - 1 : x - 1, xp = x == G.nx - 1 ? 0 : x + 1;
    auto at = [&](int p, int r, int xx) { return __ldg(a.lam_in + p * G.plane + (long long)r * G.pitch + xx); };
    const long long o = (long long)row * G.pitch + x;
    const double gacc = a.gcl[o];
    float v[21], sg[3];
#pragma unroll
    for (int g = 0; g < 3; g++) {
        v[0 + g] = at(0 + g, row, x);
        v[3 + g] = at(3 + g, row, xm);
        v[6 + g] = at(6 + g, rym, x);
        v[9 + g] = at(9 + g, rzm, x);
        v[12 + g] = at(12 + g, row, xp);
        v[15 + g] = at(15 + g, ryp, x);
        v[18 + g] = at(18 + g, rzp, x);
        sg[g] = __ldg(sig + g * G.plane + o);
    }
    const float q = __ldg(a.cL2 + o);
    AdjEvents3 ev = {};
    if (a.evt.rowptr) {
        const int e0 = __ldg(a.evt.rowptr + row), e1 = __ldg(a.evt.rowptr + row + 1);
        for (int e = e0; e < e1; e++) {
            const Event k = a.evt.ev[e];
            if (k.x == x) adjoint3_event(ev, k, a.evt, a.cot, a.nsteps, a.t, a.t0);
        }
    }
    a.gcl[o] = gacc + (double)adjoint3_site(v, sg, q, ev);
#pragma unroll
    for (int p = 0; p < 21; p++) __stcs(a.lam_out + p * G.plane + o, v[p]);
}

// dL/d eps_r = -dL/dc_L^2 * c_L^2 / eps_r with eps_r = (D-1) c_ref^2 / c_L^2 (mu = 1), dense output.
__global__ void adjoint_finish(Grid G, const double *gcl, const float *cL2, int D, double c_ref2, float *geps,
                               double *gcl_dense) {
    const long long n = (long long)G.nx * G.nrows;
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (long long)gridDim.x * blockDim.x) {
        const long long row = s / G.nx;
        const int x = (int)(s - row * G.nx);
        const double g = gcl[row * G.pitch + x];
        const double q = cL2[row * G.pitch + x];
        if (geps) geps[s] = (float)(-g * q * q / ((D - 1) * c_ref2));
        if (gcl_dense) gcl_dense[s] = g;
    }
}

static cudaError_t launch_adjoint(const lbem_t *h, const AdjArgs &a) {
    const long long warps = (long long)a.g.nrows * (a.g.nchunk_pad / 32);
    adjoint2d<<<(unsigned)((warps * 32 + BLOCK - 1) / BLOCK), BLOCK, 0, h->stream>>>(a);
    return cudaGetLastError();
}

// 3D: n steps from a.in at a.t, alternating between a.in and a.out, their sigmas to sig (unless null); *launches of them.
static cudaError_t forward_3d(const lbem_t *h, StepArgs a, int n, float *sig, int *launches) {
    const int groups = march3_ok(h, true) ? n / MARCH3_STEPS : 0, done = groups * MARCH3_STEPS;
    if (groups) {
        Adj3 r;
        r.sig = sig;
        const cudaError_t e = sig ? launch_march_3d_adj(a, r, true, groups, h->stream)
                                  : launch_march_3d(a, Walls(), groups, h->stream);
        if (e != cudaSuccess) return e;
        if (groups & 1) std::swap(a.in, a.out);
        a.t += done;
    }
    for (int k = done; k < n; k++) {
        const cudaError_t e = launch_step_3d(a, false, h->variant, h->stream, nullptr,
                                             sig ? sig + (size_t)k * 3 * a.g.plane : nullptr);
        if (e != cudaSuccess) return e;
        std::swap(a.in, a.out);
        a.t++;
    }
    *launches = groups + n - done;
    return cudaSuccess;
}

// 3D: n adjoint steps back from a.t, lambda from a.in, alternating with a.out; adj.sig: the sigma of step a.t.
static cudaError_t adjoint_sigma(const lbem_t *h, StepArgs a, Adj3 adj, int n, int *launches) {
    const int groups = march3_ok(h, true) ? n / MARCH3_STEPS : 0, done = groups * MARCH3_STEPS;
    if (groups) {
        const cudaError_t e = launch_march_3d_adj(a, adj, false, groups, h->stream);
        if (e != cudaSuccess) return e;
        if (groups & 1) std::swap(a.in, a.out);
        a.t -= done;
        adj.sig -= (long long)done * 3 * a.g.plane;
    }
    for (int k = done; k < n; k++) {
        AdjArgs q;
        q.g = a.g;
        q.lam_in = static_cast<const float *>(a.in.data);
        q.lam_out = static_cast<float *>(a.out.data);
        q.cL2 = a.med.cL2;
        q.gcl = adj.gcl;
        q.evt = a.evt;
        q.cot = adj.cot;
        q.nsteps = adj.nsteps;
        q.t = a.t;
        q.t0 = adj.t0;
        const unsigned blocks = (unsigned)(((long long)a.g.nrows * a.g.pitch + BLOCK - 1) / BLOCK);
        if (h->variant == 2) adjoint3d_site<5><<<blocks, BLOCK, 0, h->stream>>>(q, adj.sig);
        else adjoint3d_site<1><<<blocks, BLOCK, 0, h->stream>>>(q, adj.sig);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        std::swap(a.in, a.out);
        a.t--;
        adj.sig -= 3 * a.g.plane;
    }
    *launches = groups + n - done;
    return cudaSuccess;
}

bool is_device_ptr(const void *p);
lbem_status device_input(lbem_t *h, const float *p, size_t count, size_t off, const float **out);

}  // namespace lbk

using namespace lbk;

extern "C" {

lbem_status lbem_forward_record(lbem_t *h, int nsteps, int every) {
    if (!h) return fail(LBEM_ERR_ARG, "null handle");
    if (nsteps < 1 || every < 1) return fail(LBEM_ERR_ARG, "lbem_forward_record: nsteps >= 1 and checkpoint_every >= 1");
    if (!h->has_medium) return fail(LBEM_ERR_STATE, "lbem_forward_record: set a medium first");
    if (h->storage != LBEM_F32) return fail(LBEM_ERR_STATE, "lbem_forward_record: the adjoint needs LBEM_F32 storage");
    if (h->has_mu) return fail(LBEM_ERR_STATE, "lbem_forward_record: the adjoint supports uniform mu only (mu_r = NULL)");
    if (h->walls()) return fail(LBEM_ERR_STATE, "lbem_forward_record: the adjoint supports periodic boundaries only");
    if (h->disp || h->aniso)
        return fail(LBEM_ERR_STATE, "lbem_forward_record: the adjoint supports non-dispersive isotropic media only");
    const size_t state = (size_t)h->npop * h->grid.plane, sig = 3 * (size_t)h->grid.plane;
    every = std::min(every, nsteps);
    const int ncp = (nsteps + every - 1) / every;
    bool all = h->dim == 3 && sig * nsteps <= state * (ncp + every);
    if (h->adj) {  // the last run's buffers serve again if they are of this run's size (up to twice that)
        const size_t cap = all ? h->adj->seg_cap : h->adj->cps_cap, need = all ? sig * nsteps : state * ncp;
        if (h->adj->all != all || cap < need || cap > 2 * need) adjoint_free(h);
    }
    if (!h->adj) h->adj = new AdjointState();
    AdjointState *A = h->adj;
    all = all && ensure(A->seg, A->seg_cap, sig * nsteps);
    A->nsteps = nsteps;
    A->every = every;
    A->ncp = ncp;
    A->t0 = h->t;
    A->state_floats = state;
    A->sig_floats = sig;
    A->all = all;
    if (!A->all && !ensure(A->cps, A->cps_cap, A->state_floats * A->ncp)) {
        adjoint_free(h);
        return fail(LBEM_ERR_NOMEM, "lbem_forward_record: no room for the checkpoints");
    }
    if (A->all) {
        int launches = 0;
        LBEM_CUDA(forward_3d(h, step_args(h, h->cur), nsteps, A->seg, &launches));
        h->cur ^= launches & 1;
        h->t += nsteps;
        return LBEM_OK;
    }
    const size_t sb = A->state_floats * sizeof(float);
    for (int n = 0; n < nsteps; n++) {
        if (n % A->every == 0)
            LBEM_CUDA(cudaMemcpyAsync(A->cps + (size_t)(n / A->every) * A->state_floats, h->buf[h->cur].data, sb,
                                      cudaMemcpyDeviceToDevice, h->stream));
        StepArgs a = step_args(h, h->cur);
        int steps = 1, launches = 1;
        if (h->dim == 3) {
            steps = std::min(A->every, nsteps - n);
            LBEM_CUDA(forward_3d(h, a, steps, nullptr, &launches));
            n += steps - 1;
        } else {
            LBEM_CUDA(launch_step_2d(a, h->storage, false, h->variant, h->stream));
        }
        h->cur ^= launches & 1;
        h->t += steps;
    }
    return LBEM_OK;
}

lbem_status lbem_adjoint(lbem_t *h, const float *trace_cot, float *grad_eps, double *grad_cL2) {
    if (!h) return fail(LBEM_ERR_ARG, "null handle");
    AdjointState *A = h->adj;
    if (!A) return fail(LBEM_ERR_STATE, "lbem_adjoint: call lbem_forward_record first");
    if (h->nrec > 0 && h->cap < A->t0 + A->nsteps)
        return fail(LBEM_ERR_STATE, "lbem_adjoint: receiver capacity shorter than the recorded run");
    const size_t sb = A->state_floats * sizeof(float);
    const Grid &G = h->grid;
    const bool d3 = h->dim == 3;
    const size_t seg = A->all ? A->sig_floats * A->nsteps : (d3 ? A->sig_floats : A->state_floats) * A->every;
    if (!ensure(A->lam, A->lam_cap, 2 * A->state_floats) || !ensure(A->gcl, A->gcl_cap, (size_t)G.plane) ||
        !ensure(A->seg, A->seg_cap, seg) || (d3 && !A->all && !ensure(A->work, A->work_cap, 2 * A->state_floats)))
        return fail(LBEM_ERR_NOMEM, "lbem_adjoint: no room for the segment and adjoint buffers");
    const size_t ncot = (size_t)h->nrec * A->nsteps;
    if (ncot) {
        if (!trace_cot) return fail(LBEM_ERR_ARG, "lbem_adjoint: trace_cot is NULL but receivers are set");
        if (!ensure(A->cot, A->cot_cap, ncot)) return fail(LBEM_ERR_CUDA, "lbem_adjoint: no room for the cotangents");
        LBEM_CUDA(cudaMemcpyAsync(A->cot, trace_cot, ncot * sizeof(float), cudaMemcpyDefault, h->stream));
    }
    LBEM_CUDA(cudaMemsetAsync(A->lam, 0, sb, h->stream));  // lambda of the end
    LBEM_CUDA(cudaMemsetAsync(A->gcl, 0, sizeof(double) * G.plane, h->stream));
    int lc = 0;  // lam[lc] holds lambda^{t+1}
    StepArgs base = step_args(h, 0);
    if (d3) {
        const int nseg = A->all ? 1 : A->ncp;
        for (int k = nseg - 1; k >= 0; k--) {
            const int n0 = k * A->every, len = A->all ? A->nsteps : std::min(A->every, A->nsteps - n0);
            int launches = 0;
            if (!A->all) {  // recompute the segment's sigmas (sources on, no trace writes)
                StepArgs a = base;
                LBEM_CUDA(cudaMemcpyAsync(A->work, A->cps + (size_t)k * A->state_floats, sb, cudaMemcpyDeviceToDevice,
                                          h->stream));
                a.in.data = A->work;
                a.out.data = A->work + A->state_floats;
                a.evt.cap = 0;
                a.t = A->t0 + n0;
                LBEM_CUDA(forward_3d(h, a, len, A->seg, &launches));
            }
            StepArgs a = base;
            a.in.data = A->lam + (size_t)lc * A->state_floats;
            a.out.data = A->lam + (size_t)(lc ^ 1) * A->state_floats;
            a.t = A->t0 + n0 + len - 1;
            Adj3 q;
            q.sig = A->seg + (size_t)(len - 1) * A->sig_floats;
            q.gcl = A->gcl;
            q.cot = A->cot;
            q.nsteps = A->nsteps;
            q.t0 = A->t0;
            LBEM_CUDA(adjoint_sigma(h, a, q, len, &launches));
            lc ^= launches & 1;
        }
    }
    for (int k = d3 ? -1 : A->ncp - 1; k >= 0; k--) {
        const int n0 = k * A->every;
        const int len = std::min(A->every, A->nsteps - n0);
        LBEM_CUDA(cudaMemcpyAsync(A->seg, A->cps + (size_t)k * A->state_floats, sb, cudaMemcpyDeviceToDevice, h->stream));
        for (int j = 1; j < len; j++) {  // recompute the segment's states (sources on, no trace writes)
            StepArgs a = base;
            a.in.data = A->seg + (size_t)(j - 1) * A->state_floats;
            a.out.data = A->seg + (size_t)j * A->state_floats;
            a.evt.cap = 0;
            a.t = A->t0 + n0 + j - 1;
            LBEM_CUDA(launch_step_2d(a, h->storage, false, h->variant, h->stream));
        }
        for (int j = len - 1; j >= 0; j--) {
            AdjArgs a;
            a.g = G;
            a.lam_in = A->lam + (size_t)lc * A->state_floats;
            a.lam_out = A->lam + (size_t)(lc ^ 1) * A->state_floats;
            a.state = base.in;
            a.state.data = A->seg + (size_t)j * A->state_floats;
            a.cL2 = h->cL2;
            a.gcl = A->gcl;
            a.evt = base.evt;
            a.cot = A->cot;
            a.nsteps = A->nsteps;
            a.t = A->t0 + n0 + j;
            a.t0 = A->t0;
            LBEM_CUDA(launch_adjoint(h, a));
            lc ^= 1;
        }
    }
    const bool eh = grad_eps && !is_device_ptr(grad_eps);
    const bool ch = grad_cL2 && !is_device_ptr(grad_cL2);
    if (eh && !A->gout) LBEM_CUDA(cudaMalloc((void **)&A->gout, sizeof(float) * h->nsite));
    if (ch && !A->gcl_out) LBEM_CUDA(cudaMalloc((void **)&A->gcl_out, sizeof(double) * h->nsite));
    float *ge = eh ? A->gout : grad_eps;
    double *gc = ch ? A->gcl_out : grad_cL2;
    adjoint_finish<<<1024, 256, 0, h->stream>>>(G, A->gcl, h->cL2, h->dim, h->c_ref2, ge, gc);
    LBEM_CUDA(cudaGetLastError());
    if (eh) LBEM_CUDA(cudaMemcpyAsync(grad_eps, ge, sizeof(float) * h->nsite, cudaMemcpyDeviceToHost, h->stream));
    if (ch) LBEM_CUDA(cudaMemcpyAsync(grad_cL2, gc, sizeof(double) * h->nsite, cudaMemcpyDeviceToHost, h->stream));
    if (eh || ch) LBEM_CUDA(cudaStreamSynchronize(h->stream));
    return LBEM_OK;
}

}  // extern "C"
