// trtr_adjoint.cu -- discrete adjoint of the TRT-R step (Eq. (14)) for gradients of a
// function J of the final phi with respect to the diffusivity field D(x).
//
// Forward (trtr_forward_record): n steps of the ordinary step kernel, keeping a copy of
// the state every k steps (k = ceil(sqrt(n)) by default).  Backward (trtr_adjoint): for
// each segment, last to first, the segment's states are recomputed from its checkpoint into
// a pool by the step kernels; then one backward kernel per step runs from the segment's end
// to its start.  Total work: two forward sweeps and one
// backward sweep; memory: about 2 sqrt(n) states.
//
// Notation (lattice units, S = 0).  The stored array holds P_i(x) = post_i(g(x)) with
// g_i(x) = P_i(x - e_i); Q_i(x) = dJ/dP_i(x).  Per node the step is
//   raw moments (phi, j, Pi) of g  ->  Hermite coefficients c  ->  post = R c,
//   c0 = phi, c1 = (1-k1) phi u + kh phi a + k1 j, c2 = (1-k2) phi (u u - 1/3 I) + k2 Pi,
//   c3 = phi (u_x^2 u_y, u_x u_y^2),  post_i = w_i [c0 + 3 e.c1 + 4.5 H2_i:c2 + 13.5 H3_i.c3],
// with k1 = 1 - 1/tau1, kh = 1 - 1/(2 tau1), k2 = 1 - 1/tau2.  Hence, with mu = Q^{n+1}(x):
//   r = R^T mu  (r0 = sum w mu, r1 = 3 sum w mu e, r2 = 4.5 sum w mu H2, r3 = 13.5 sum w mu H3),
//   lambda^n_i(x) = dJ/dg^n_i(x) = [moments^T  relax^T  r]_i,   Q^n_i(x - e_i) = lambda^n_i(x),
//   dJ/dD(x) += dtau1/dD [ r1 . dc1/dtau1 + dtau2/dtau1  r2 : dc2/dtau2 ],
//   dc1/dtau1 = (j - phi u)/tau1^2 + phi a/(2 tau1^2),   dc2/dtau2 = (Pi - phi/3 I - phi u u)/tau2^2,
//   dtau1/dD = 3 dt/dx^2,  dtau2/dtau1 = -Lambda/(tau1 - 1/2)^2 (magic) or 0 (fixed tau2).
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <new>
#include <type_traits>
#include <vector>

#include "trtr_step_core.cuh"
#include "trtr_trace.h"

struct trtr_adjoint_state {
    long n0, steps;
    int interval, nseg;
    size_t state_bytes;
    std::vector<void*> ckpt;
    std::vector<void*> pool;
    std::vector<CUtensorMap> pool_maps;
    std::vector<CUtensorMap> pool_maps2;  // the two-step kernel's maps of the pool
    std::vector<CUtensorMap> ckpt_maps, ckpt_maps2;  // of the checkpoints (a segment's first state)
    bool two;                             // the recomputation takes pairs of steps per launch
    void* Q[2];
    double* grad;
    void* fields;  // packed fields of a context without the two-step kernel's (FP32-computing storages)
    trtr::PlaneLayout lq;
};

namespace trtr {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ int wrapi(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

template <typename C>
__global__ void adj_init_kernel(C* Q, const double* dJ, PlaneLayout lq) {
    // Q_i(x) = dJ/dP_i(x) = dJ/dg^N_i(x + e_i) = dJ/dphi(x + e_i)
    const unsigned n = (unsigned)lq.nx * lq.ny;
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int j = (int)(k / lq.nx), i = (int)(k - (unsigned)j * lq.nx);
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const int si = wrapi(i + lattice_ex(q), lq.nx), sj = wrapi(j + lattice_ey(q), lq.ny);
            Q[q * lq.plane + lq.at(i, j)] = C(dJ[(size_t)sj * lq.nx + si]);
        }
    }
}

using core::F2;
using core::vfma;
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double divide(double a, double b) { return a / b; }
__device__ __forceinline__ F2 divide(F2 a, F2 b) { return F2(a.v.x / b.v.x, a.v.y / b.v.y); }

// The transpose of one node's step, and the node's gradient terms.  Q: dJ/dP^{n+1}, g: the
// pre-collision populations (D only).  Returns lambda^n; d1 = r1 . dc1/dtau1, d2 = r2 : dc2/dtau2 and
// dtau2_dtau1 (Eq. (28)).  r = R^T Q is taken from the sums and differences of opposite directions
// with the weights folded in, and lambda is rebuilt pairwise: about 110 operations in all.
template <typename V, bool D>
__device__ __forceinline__ void adjoint_node(const V Q[kQ], const V g[kQ], V ux, V uy, V ax, V ay, V w1, V w2, V lam[kQ],
                                             V& d1, V& d2) {
    using T = std::conditional_t<std::is_same<V, double>::value, double, float>;
    const V k1 = V(T(1)) - w1, k2 = V(T(1)) - w2, kh = vfma(V(T(-0.5)), w1, V(T(1)));
    const V s12 = Q[1] + Q[2], s34 = Q[3] + Q[4], s56 = Q[5] + Q[6], s78 = Q[7] + Q[8];
    const V d12 = Q[1] - Q[2], d34 = Q[3] - Q[4], d56 = Q[5] - Q[6], d78 = Q[7] - Q[8];
    const V ds = d56 + d78, dd = d56 - d78, sd = s56 + s78;
    const V r0 = vfma(V(T(4.0 / 9.0)), Q[0], vfma(V(T(1.0 / 9.0)), s12 + s34, V(T(1.0 / 36.0)) * sd));
    const V r1x = vfma(V(T(1.0 / 3.0)), d12, V(T(1.0 / 12.0)) * ds);
    const V r1y = vfma(V(T(1.0 / 3.0)), d34, V(T(1.0 / 12.0)) * dd);
    const V t = vfma(V(T(0.125)), sd, V(T(-1.5)) * r0);
    const V rxx = vfma(V(T(0.5)), s12, t), ryy = vfma(V(T(0.5)), s34, t), rxy = V(T(0.25)) * (s56 - s78);
    const V r3a = vfma(V(T(0.375)), dd, V(T(-1.5)) * r1y), r3b = vfma(V(T(0.375)), ds, V(T(-1.5)) * r1x);

    // relax^T r: the adjoints of the raw moments
    const V second = vfma(vfma(rxx, ux, rxy * uy), ux, (ryy * uy) * uy);
    const V third = (ux * uy) * vfma(r3a, ux, r3b * uy);
    V nphi = vfma(r1x, vfma(w1, ux, kh * ax), vfma(r1y, vfma(w1, uy, kh * ay), r0));
    nphi = vfma(w2, second, nphi) + third;
    nphi = vfma(V(T(-1.0 / 3.0)) * k2, rxx + ryy, nphi);
    const V njx = k1 * r1x, njy = k1 * r1y, nxx = k2 * rxx, nyy = k2 * ryy, nxy = k2 * rxy;

    const V ex = nphi + nxx, ey = nphi + nyy, ed = ex + nyy, ep = ed + nxy, em = ed - nxy, op = njx + njy, om = njx - njy;
    lam[0] = nphi;
    lam[1] = ex + njx;
    lam[2] = ex - njx;
    lam[3] = ey + njy;
    lam[4] = ey - njy;
    lam[5] = ep + op;
    lam[6] = ep - op;
    lam[7] = em + om;
    lam[8] = em - om;

    if constexpr (D) {
        const V p12 = g[1] + g[2], p34 = g[3] + g[4], p56 = g[5] + g[6], p78 = g[7] + g[8], pd = p56 + p78;
        const V e56 = g[5] - g[6], e78 = g[7] - g[8];
        const V pxx = p12 + pd, pyy = p34 + pd, pxy = p56 - p78;
        const V phi = (g[0] + pxx) + p34;
        const V jx = (g[1] - g[2]) + (e56 + e78), jy = (g[3] - g[4]) + (e56 - e78);
        const V px = phi * ux, py = phi * uy, h = V(T(0.5)) * phi, th = V(T(1.0 / 3.0)) * phi;
        const V b1x = vfma(h, ax, jx - px), b1y = vfma(h, ay, jy - py);
        d1 = (w1 * w1) * vfma(r1x, b1x, r1y * b1y);
        const V bxx = (pxx - th) - px * ux, byy = (pyy - th) - py * uy, bxy = pxy - px * uy;
        d2 = (w2 * w2) * vfma(rxx, bxx, vfma(ryy, byy, rxy * bxy));
    }
}

struct AdjArgs {
    PlaneLayout lp, lf, lq;  // populations; fields (FP32: packed u, a, D; FP64: u, a and D apart); adjoints
    float phi_ref;
    int tau2_fixed;
    double magic, w2_fixed, dtau1_dD;
};

// One step backwards: lambda of every node from Qin, stored pushed back, Q^n_q(x - e_q) = lambda_q(x),
// and the gradient's share.  FP32-computing storages take a node pair per thread (packed
// arithmetic), FP64 a node.  The recorded state and the fields are loaded before the wait for the
// launch before this one: a launch lets the next one start only after its own wait, so everything but
// the last launch has then completed, and that writes adjoints and the gradient alone.
// Measured (GB300, 512^2 FP32): 11.5 us with one node a thread, the velocity stencil and the wrapped
// stores of every node; see launch_adjoint_step.
template <typename S, typename C, bool D>
__global__ void __launch_bounds__(kThreads)
    adj_step_kernel(const S* __restrict__ P, const C* Qin, C* Qout, double* grad, const C* __restrict__ fields,
                    const C* __restrict__ accel, const C* __restrict__ Dh, const AdjArgs a) {
    constexpr bool kF64 = sizeof(S) == 8;
    using V = std::conditional_t<kF64, double, F2>;
    constexpr int kN = kF64 ? 1 : 2;  // nodes a thread
    const int nx = a.lp.nx, ny = a.lp.ny;
    const unsigned per = (nx + kN - 1) / kN, n = per * (unsigned)ny;
    const unsigned k = blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = k < n;
    const int j = in ? (int)(k / per) : 0, i = in ? kN * (int)(k - (unsigned)j * per) : 0;
    const bool ok = in_frame(a.lp, i - 1, j - 1, 1, 1) && in_frame(a.lp, i + kN, j + 1, kN, 1) &&
                    in_frame(a.lf, i + kN - 1, j, 1, 0) && in_frame(a.lq, i + kN - 1, j, 1, 0);
    V g[kQ], ux, uy, ax, ay, w1, w2, dt2;
    if (in && ok) {
        const size_t at = a.lp.at(i, j), o = a.lf.at(i, j), pl = a.lf.plane;
#pragma unroll
        for (int q = 0; q < kQ; ++q) {  // pull (the ghost cells hold the periodic images)
            if constexpr (!D) {
                g[q] = V(0.f);
            } else {
                const S* p = P + q * a.lp.plane + at - (ptrdiff_t)lattice_ey(q) * a.lp.pitch - lattice_ex(q);
                if constexpr (kF64) {
                    g[q] = p[0];
                } else {
                    const float off = core::weight<float>(q) * a.phi_ref;
                    g[q] = lattice_ex(q) == 0
                               ? core::Pair<S>::decode(*reinterpret_cast<const typename core::Pair<S>::type*>(p), off)
                               : core::Pair<S>::decode(p[0], p[1], off);
                }
            }
        }
        auto field = [&](const C* f) {
            if constexpr (kF64)
                return f[o];
            else
                return F2(*reinterpret_cast<const float2*>(f + o));
        };
        ux = field(fields);
        uy = field(fields + pl);
        ax = field(accel);
        ay = field(accel + pl);
        // tau1 - 1/2 = 3 D (Sec. 2.4); tau2 from Lambda (Eq. (28)) or fixed
        using T = std::conditional_t<kF64, double, float>;
        const V t1m = V(T(3)) * field(Dh), magic((T)a.magic);
        w1 = divide(V(T(1)), V(T(0.5)) + t1m);
        w2 = a.tau2_fixed ? V((T)a.w2_fixed) : divide(t1m, vfma(V(T(0.5)), t1m, magic));
        dt2 = a.tau2_fixed ? V(T(0)) : divide(V(T(-1)) * magic, t1m * t1m);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (!in || !ok) return;
    V Q[kQ], lam[kQ], d1, d2;
    const size_t aq = a.lq.at(i, j);
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        if constexpr (kF64)
            Q[q] = Qin[q * a.lq.plane + aq];
        else
            Q[q] = F2(*reinterpret_cast<const float2*>(Qin + q * a.lq.plane + aq));
    }
    adjoint_node<V, D>(Q, g, ux, uy, ax, ay, w1, w2, lam, d1, d2);
    const bool inner = i >= 1 && i + kN < nx && j >= 1 && j + 1 < ny;
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        C* plane = Qout + q * a.lq.plane;
        auto put = [&](int ii, C v) {
            plane[a.lq.at(wrapi(ii - lattice_ex(q), nx), wrapi(j - lattice_ey(q), ny))] = v;
        };
        if constexpr (kF64) {
            put(i, lam[q]);
        } else if (inner) {
            if (!in_frame(a.lq, i - lattice_ex(q), j - lattice_ey(q), 0, 0) || !in_frame(a.lq, i + 1 - lattice_ex(q), j, 0, 0)) continue;
            C* p = plane + aq - (ptrdiff_t)lattice_ey(q) * a.lq.pitch - lattice_ex(q);
            if (lattice_ex(q) == 0) {
                *reinterpret_cast<float2*>(p) = lam[q].v;
            } else {
                p[0] = lam[q].v.x;
                p[1] = lam[q].v.y;
            }
        } else {
            put(i, lam[q].v.x);
            if (i + 1 < nx) put(i + 1, lam[q].v.y);
        }
    }
    if constexpr (D) {
        double* gp = grad + (size_t)j * nx + i;
        if constexpr (kF64) {
            gp[0] = fma(a.dtau1_dD, fma(dt2, d2, d1), gp[0]);
        } else {
            // d1 + dtau2/dtau1 d2 as the sum of two floats (exact product, error-free sum): two conversions
            // to the slow FP64 pipe instead of three and a product
            const F2 p = dt2 * d2, pe = vfma(dt2, d2, F2(0.f) - p);
            const F2 s = d1 + p, bb = s - d1, lo = ((d1 - (s - bb)) + (p - bb)) + pe;
            gp[0] = fma(a.dtau1_dD, (double)s.v.x + (double)lo.v.x, gp[0]);
            if (i + 1 < nx) gp[1] = fma(a.dtau1_dD, (double)s.v.y + (double)lo.v.y, gp[1]);
        }
    }
}

int grid_for(const trtr_ctx* ctx) {
    const size_t n = (size_t)ctx->p.nx * ctx->p.ny;
    const size_t want = (n + kThreads - 1) / kThreads, cap = (size_t)ctx->num_sms * 8;
    return (int)(want < 1 ? 1 : (want > cap ? cap : want));
}

int adj_csize(const trtr_ctx* ctx) { return ctx->p.precision == TRTR_F64 ? 8 : 4; }

// One adjoint step from the recorded state P.  alone: it starts after the launch before it has
// completed (the first of a segment, whose state that launch may write).
template <typename S, typename C>
cudaError_t launch_adjoint_typed(trtr_ctx* ctx, const void* P, const void* Qin, void* Qout, const void* fields, bool alone) {
    const trtr_adjoint_state* s = ctx->adj;
    constexpr bool kF64 = sizeof(S) == 8;
    AdjArgs a;
    a.lp = ctx->lp;
    a.lf = kF64 ? ctx->lf : ctx->lt;
    a.lq = s->lq;
    a.phi_ref = (float)ctx->p.phi_ref;
    a.tau2_fixed = ctx->p.tau2_mode == TRTR_TAU2_FIXED;
    a.magic = ctx->p.magic;
    a.w2_fixed = a.tau2_fixed ? 1.0 / ctx->p.tau2 : 0.0;
    a.dtau1_dD = 3.0 * ctx->p.dt / (ctx->p.dx * ctx->p.dx);
    const C* f = static_cast<const C*>(fields);
    const C* accel = kF64 ? static_cast<const C*>(ctx->pack64) : f + 2 * ctx->lt.plane;
    const C* D = kF64 ? static_cast<const C*>(ctx->Dh) : f + 4 * ctx->lt.plane;
    const size_t n = (size_t)(kF64 ? ctx->p.nx : (ctx->p.nx + 1) / 2) * ctx->p.ny;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((n + kThreads - 1) / kThreads));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = !alone;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const S* p = static_cast<const S*>(P);
    const C* qi = static_cast<const C*>(Qin);
    C* qo = static_cast<C*>(Qout);
    const bool d_enters = !(ctx->p.tau1_const > 0.0);
    return d_enters ? cudaLaunchKernelEx(&cfg, adj_step_kernel<S, C, true>, p, qi, qo, s->grad, f, accel, D, a)
                    : cudaLaunchKernelEx(&cfg, adj_step_kernel<S, C, false>, p, qi, qo, s->grad, f, accel, D, a);
}

cudaError_t launch_adjoint_step(trtr_ctx* ctx, const void* P, const void* Qin, void* Qout, const void* fields, bool alone) {
    switch (ctx->p.precision) {
        case TRTR_F64: return launch_adjoint_typed<double, double>(ctx, P, Qin, Qout, fields, alone);
        case TRTR_F32: return launch_adjoint_typed<float, float>(ctx, P, Qin, Qout, fields, alone);
        case TRTR_F16_OFS: return launch_adjoint_typed<__half, float>(ctx, P, Qin, Qout, fields, alone);
        case TRTR_BF16_OFS: return launch_adjoint_typed<__nv_bfloat16, float>(ctx, P, Qin, Qout, fields, alone);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// The fields that the adjoint step reads, packed if u or D changed since they were.
cudaError_t ensure_adjoint_fields(trtr_ctx* ctx, const void** fields) {
    cudaError_t e = cudaSuccess;
    if (ctx->p.precision == TRTR_F64) {
        *fields = ctx->uv;
        if (!ctx->pack64_ready) e = launch_pack_f64(ctx);
        ctx->pack64_ready = e == cudaSuccess;
    } else if (ctx->fld2) {
        *fields = ctx->fld2;
        if (!ctx->fld2_ready) e = launch_pack_fields2(ctx);
        ctx->fld2_ready = e == cudaSuccess;
    } else {
        *fields = ctx->adj->fields;
        e = launch_pack_fields2_into(ctx, ctx->adj->fields);
    }
    return e;
}

void free_adjoint(trtr_ctx* ctx) {
    trtr_adjoint_state* a = ctx->adj;
    if (!a) return;
    cudaStreamSynchronize(ctx->stream);
    for (void* p : a->ckpt) cudaFree(p);
    for (void* p : a->pool) cudaFree(p);
    if (a->Q[0]) cudaFree(a->Q[0]);
    if (a->Q[1]) cudaFree(a->Q[1]);
    if (a->grad) cudaFree(a->grad);
    if (a->fields) cudaFree(a->fields);
    cudaGetLastError();
    delete a;
    ctx->adj = nullptr;
}

TRTR_BOUNDS_TAKE(adjoint)

}  // namespace trtr

namespace {

trtr_status adj_fail(trtr_ctx* ctx, trtr_status s, const char* msg) {
    snprintf(ctx->err, sizeof(ctx->err), "%s", msg);
    return s;
}

}  // namespace

extern "C" {

trtr_status trtr_forward_record(trtr_ctx* ctx, long steps, int interval) {
    trtr::TraceRange trace("trtr_forward_record");
    if (!ctx) return TRTR_EINVAL;
    if (steps < 1 || interval < 0) return adj_fail(ctx, TRTR_EINVAL, "steps >= 1 and interval >= 0 required");
    if (!ctx->initialized) return adj_fail(ctx, TRTR_ESTATE, "populations not initialised");
    if (ctx->p.src_mode != TRTR_SRC_NONE) return adj_fail(ctx, TRTR_EINVAL, "the adjoint supports S = 0 only");
    if (ctx->p.bc_mode != TRTR_BC_PERIODIC)
        return adj_fail(ctx, TRTR_EINVAL, "the adjoint supports periodic boundaries only");
    const int every = interval > 0 ? (interval < steps ? interval : (int)steps) : (int)ceil(sqrt((double)steps));
    const int nseg = (int)((steps + every - 1) / every);
    const bool two = trtr::two_step_applies(ctx);
    // the buffers of the record before this one are kept where its checkpoints are as many and as far
    // apart: 30 allocations and releases took 2.4 of the 7.4 ms of a 200-step gradient at 512^2
    trtr_adjoint_state* a = ctx->adj;
    if (a && (a->interval != every || a->nseg != nseg || a->two != two)) {
        trtr::free_adjoint(ctx);
        a = nullptr;
    }
    if (a) {
        a->n0 = ctx->step;
        a->steps = steps;
    } else {
        a = new (std::nothrow) trtr_adjoint_state();
        if (!a) return TRTR_ENOMEM;
        ctx->adj = a;
        a->n0 = ctx->step;
        a->steps = steps;
        a->interval = every;
        a->nseg = nseg;
        a->two = two;
        a->state_bytes = trtr::kQ * ctx->lp.plane * ctx->esize;
        a->lq = trtr::make_layout(ctx->p.nx, ctx->p.ny, trtr::adj_csize(ctx), 1);
        const size_t qbytes = trtr::kQ * a->lq.plane * trtr::adj_csize(ctx);
        const bool pack = ctx->p.precision != TRTR_F64 && !ctx->fld2;
        bool ok = cudaMalloc(&a->Q[0], qbytes) == cudaSuccess && cudaMalloc(&a->Q[1], qbytes) == cudaSuccess &&
                  cudaMalloc(&a->grad, (size_t)ctx->p.nx * ctx->p.ny * sizeof(double)) == cudaSuccess &&
                  (!pack || cudaMalloc(&a->fields, 5 * ctx->lt.plane * sizeof(float)) == cudaSuccess);
        auto state = [&](std::vector<void*>& v, std::vector<CUtensorMap>& maps, std::vector<CUtensorMap>& maps2) {
            void* p = nullptr;
            ok = ok && cudaMalloc(&p, a->state_bytes) == cudaSuccess;
            if (!ok) return;
            v.push_back(p);
            CUtensorMap m = {};
            ok = trtr::encode_pop_map(ctx, p, &m) == cudaSuccess;
            maps.push_back(m);
            if (ok && two) {
                ok = trtr::encode_pop_map2(ctx, p, &m) == cudaSuccess;
                maps2.push_back(m);
            }
        };
        for (int s = 0; ok && s < nseg; ++s) state(a->ckpt, a->ckpt_maps, a->ckpt_maps2);
        for (int s = 0; ok && s < every; ++s) state(a->pool, a->pool_maps, a->pool_maps2);
        if (!ok) {
            cudaGetLastError();
            trtr::free_adjoint(ctx);
            return adj_fail(ctx, TRTR_ENOMEM, "cannot allocate the checkpoints of the adjoint");
        }
    }
    // the recorded run keeps only the checkpoint states, so several steps between two checkpoints may
    // run as one launch (the same states bit for bit)
    trtr::begin_steps(ctx);
    const char* what = "";
    for (long k = 0; k < steps;) {
        what = "checkpoint copy";
        if (k % a->interval == 0 &&
            cudaMemcpyAsync(a->ckpt[k / a->interval], ctx->pop[ctx->cur], a->state_bytes, cudaMemcpyDeviceToDevice,
                            ctx->stream) != cudaSuccess)
            break;
        const long to_checkpoint = a->interval - k % a->interval;
        int taken = 0;
        if (trtr::launch_steps(ctx, to_checkpoint < steps - k ? to_checkpoint : steps - k, steps, &taken, &what) != cudaSuccess)
            break;
        k += taken;
        what = nullptr;
    }
    trtr::end_steps(ctx);
    return what ? adj_fail(ctx, TRTR_ECUDA, what) : TRTR_OK;
}

trtr_status trtr_adjoint(trtr_ctx* ctx, const double* dJ_dphi, int on_device, double* grad_D, int grad_on_device) {
    trtr::TraceRange trace("trtr_adjoint");
    if (!ctx) return TRTR_EINVAL;
    if (!dJ_dphi || !grad_D) return adj_fail(ctx, TRTR_EINVAL, "dJ_dphi and grad_D are required");
    trtr_adjoint_state* a = ctx->adj;
    if (!a || ctx->step != a->n0 + a->steps)
        return adj_fail(ctx, TRTR_ESTATE, "no recorded forward run ending at the current step");
    const size_t n = (size_t)ctx->p.nx * ctx->p.ny;
    cudaStream_t st = ctx->stream;
    const double* dJ = dJ_dphi;
    double* stage = nullptr;
    if (!on_device) {
        if (cudaMalloc(&stage, n * sizeof(double)) != cudaSuccess) return TRTR_ENOMEM;
        if (cudaMemcpyAsync(stage, dJ_dphi, n * sizeof(double), cudaMemcpyHostToDevice, st) != cudaSuccess) {
            cudaFree(stage);
            return TRTR_ECUDA;
        }
        dJ = stage;
    }
    cudaError_t e = cudaMemsetAsync(a->grad, 0, n * sizeof(double), st);
    const int grid = trtr::grid_for(ctx);
    if (e == cudaSuccess) {
        if (ctx->p.precision == TRTR_F64)
            trtr::adj_init_kernel<double><<<grid, trtr::kThreads, 0, st>>>((double*)a->Q[0], dJ, a->lq);
        else
            trtr::adj_init_kernel<float><<<grid, trtr::kThreads, 0, st>>>((float*)a->Q[0], dJ, a->lq);
        e = cudaGetLastError();
    }
    // the packed fields, if u or D changed since they were packed
    const void* fields = nullptr;
    if (e == cudaSuccess) e = trtr::ensure_adjoint_fields(ctx, &fields);
    int qc = 0;
    for (int seg = a->nseg - 1; seg >= 0 && e == cudaSuccess; --seg) {
        const long s0 = (long)seg * a->interval;
        const long len = a->steps - s0 < a->interval ? a->steps - s0 : a->interval;
        // recompute the segment's states from its checkpoint: pairs through the two-step kernel, which
        // stores the intermediate state as well (the checkpoint may carry only the one-wide ghost frame,
        // so its outer ring is refreshed first), a last odd step by the one-step kernel
        const bool pairs = a->two && len >= 3;
        auto buffer = [&](long k) { return k == 0 ? a->ckpt[seg] : a->pool[k]; };
        if (pairs && e == cudaSuccess) e = trtr::launch_refresh_ghosts2_buffer(ctx, buffer(0));
        long recompute_launches = 0;
        for (long k = 0; k + 1 < len && e == cudaSuccess; ++recompute_launches) {
            if (pairs && k + 2 < len) {
                e = trtr::launch_step2_from(ctx, k == 0 ? &a->ckpt_maps2[seg] : &a->pool_maps2[k], a->pool[k + 2],
                                            a->pool[k + 1], a->n0 + s0 + k);
                k += 2;
            } else {
                e = trtr::launch_step_from(ctx, buffer(k), k == 0 ? &a->ckpt_maps[seg] : &a->pool_maps[k], a->pool[k + 1],
                                           a->n0 + s0 + k);
                k += 1;
            }
        }
        for (long k = len - 1; k >= 0 && e == cudaSuccess; --k) {
            e = trtr::launch_adjoint_step(ctx, buffer(k), a->Q[qc], a->Q[qc ^ 1], fields, k == len - 1);
            qc ^= 1;
        }
        ctx->launches += recompute_launches + len;  // the recomputation and the adjoint steps
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(grad_D, a->grad, n * sizeof(double),
                            grad_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, st);
    cudaError_t es = cudaStreamSynchronize(st);
    if (stage) cudaFree(stage);
    if (e != cudaSuccess || es != cudaSuccess) {
        cudaGetLastError();
        return adj_fail(ctx, TRTR_ECUDA, cudaGetErrorString(e != cudaSuccess ? e : es));
    }
    return TRTR_OK;
}

}  // extern "C"
