// trtr_f64.cu -- the FP64 time step of the evolution equation (14): one launch per step, one node
// per thread.
//
// What bounds it: the FP64 pipe.  An SM takes 16 cycles for an FP64 warp instruction (2 lanes a
// cycle), so a node's arithmetic costs what 30 times its bytes would, and the step is planned to
// take few FP64 instructions and to give every SM its share of them:
//  - what does not change from step to step is packed once per change of the fields, four planes
//    beside u: the acceleration a = (u . grad) u and the relaxation factors k1 = 1 - 1/tau1,
//    k2 = 1 - 1/tau2 (two divisions and the eight differences a node);
//  - the update takes 72 FP64 instructions (81 with a source);
//  - nodes are numbered through the rows, so only the last warp is ragged, and small grids run in
//    blocks of one warp, spread over all SMs (in tiles of 64 x 8 nodes a 64^2 grid kept 8 of 152 SMs
//    busy).
// Plain loads are enough: at 8 GLUPS the step moves 1.7 TB/s.  Measured (GB300): see launch_step_f64.
#include "trtr_step_core.cuh"

namespace trtr {
namespace {

using namespace core;

struct F64Args {
    const double* src;
    double* dst;
    const double* uv;     // [2][rows][pitch]
    const double* pack;   // [4][rows][pitch]: a_x, a_y, k1, k2 (the layout of uv)
    const double* s_n;    // source planes (TRTR_SRC_FIELD)
    const double* s_p;
    const double* pulse;  // tables of level n - 1 (TRTR_SRC_PULSE)
    PulseTab pt;
    PlaneLayout lp, lf;
};

// The node update in moment space, as collide_node (trtr_step_core.cuh) with the constant factors
// given and the diagonal pairs rebuilt from P = m1x/3 + T_xyy, Q = m1y/3 + T_xxy:
// their odd parts are (P + Q)/4 and (P - Q)/4.
template <bool SOURCE>
__device__ __forceinline__ void collide_f64(const double g[kQ], double ux, double uy, double ax, double ay, double k1,
                                            double k2, double s, double out[kQ]) {
    const double p12 = g[1] + g[2], p34 = g[3] + g[4], p56 = g[5] + g[6], p78 = g[7] + g[8];
    const double d12 = g[1] - g[2], d34 = g[3] - g[4], d56 = g[5] - g[6], d78 = g[7] - g[8];
    const double pd = p56 + p78, pxx = p12 + pd, pyy = p34 + pd, pxy = p56 - p78;
    const double phi = (g[0] + pxx) + p34;
    const double jx = d12 + (d56 + d78), jy = d34 + (d56 - d78);
    const double phux = phi * ux, phuy = phi * uy;
    const double euxx = phux * ux, euyy = phuy * uy, euxy = phux * uy;
    const double kh = fma(0.5, k1, 0.5);  // 1 - 1/(2 tau1)
    const double m0 = SOURCE ? phi + s : phi;
    const double hx = SOURCE ? fma(phi, ax, ux * s) : phi * ax, hy = SOURCE ? fma(phi, ay, uy * s) : phi * ay;
    const double X = (1.0 / 3.0) * fma(kh, hx, fma(k1, jx - phux, phux));
    const double Y = (1.0 / 3.0) * fma(kh, hy, fma(k1, jy - phuy, phuy));
    const double third = phi * (1.0 / 3.0);
    const double Axx = fma(k2, (pxx - third) - euxx, euxx), Ayy = fma(k2, (pyy - third) - euyy, euyy);
    const double Axy = fma(k2, pxy - euxy, euxy);
    const double Txxy = euxx * uy, Txyy = euxy * uy;
    const double P = X + Txyy, Q = Y + Txxy, sum = P + Q, dif = P - Q;
    const double O1 = fma(-0.5, Txyy, X), O3 = fma(-0.5, Txxy, Y);
    const double As = Axx + Ayy, m9 = m0 * (1.0 / 9.0), c = fma(-1.0 / 6.0, As, m9);
    const double E1 = fma(0.5, Axx, c), E3 = fma(0.5, Ayy, c);
    const double Ed = fma(1.0 / 12.0, As, 0.25 * m9);
    const double E5 = fma(0.25, Axy, Ed), E7 = fma(-0.25, Axy, Ed);
    out[1] = E1 + O1;
    out[2] = E1 - O1;
    out[3] = E3 + O3;
    out[4] = E3 - O3;
    out[5] = fma(0.25, sum, E5);
    out[6] = fma(-0.25, sum, E5);
    out[7] = fma(0.25, dif, E7);
    out[8] = fma(-0.25, dif, E7);
    // the rest population closes the mass balance (collide_node)
    out[0] = fma(-2.0, E1, fma(-2.0, E3, fma(-2.0, E5, fma(-2.0, E7, m0))));
}

template <int SRC>
__global__ void __launch_bounds__(128) f64_step_kernel(const __grid_constant__ F64Args a) {
    const unsigned k = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned nx = a.lp.nx, ny = a.lp.ny;
    const bool in = k < nx * ny;
    const unsigned j = k / nx, i = k - j * nx;
    // What earlier steps do not write is loaded while they may still run (programmatic dependent launch).  The next
    // launch may come from the wait on: let in at the start, several launches' blocks waited side by side and a
    // launch's own blocks went to the SMs that had room, a few of the 152 (us a step: 16 x 2000 20.9, now 6.7;
    // 1000 x 33 21.2, now 6.5; 130^2 8.2, now 4.6; 64^2 4.4, now 4.2).
    double ux = 0, uy = 0, ax = 0, ay = 0, k1 = 0, k2 = 0, s = 0;
    if (in) {
        const size_t o = a.lf.at_g<kGhostF>(i, j), pl = a.lf.plane;
        ux = __ldg(a.uv + o);
        uy = __ldg(a.uv + pl + o);
        ax = __ldg(a.pack + o);
        ay = __ldg(a.pack + pl + o);
        k1 = __ldg(a.pack + 2 * pl + o);
        k2 = __ldg(a.pack + 3 * pl + o);
        if (SRC == TRTR_SRC_PULSE) s = pulse_source_dt(a.pulse, a.pt, i, j);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (!in) return;
    double g[kQ], out[kQ];
    const size_t at = a.lp.at_g<kGhostP>(i, j);
    if (!in_frame(a.lp, (int)i - 1, (int)j - 1, 1, 1) || !in_frame(a.lp, (int)i + 1, (int)j + 1, 1, 1)) return;
#pragma unroll
    for (int q = 0; q < kQ; ++q)
        g[q] = a.src[q * a.lp.plane + at - (ptrdiff_t)lattice_ey(q) * a.lp.pitch - lattice_ex(q)];
    if (SRC == TRTR_SRC_FIELD) {
        const size_t o = a.lf.at_g<kGhostF>(i, j);
        s = fma(1.5, a.s_n[o], -0.5 * a.s_p[o]);
    }
    collide_f64<SRC != TRTR_SRC_NONE>(g, ux, uy, ax, ay, k1, k2, s, out);
    if (i >= 1 && i + 1 < nx && j >= 1 && j + 1 < ny) {
#pragma unroll
        for (int q = 0; q < kQ; ++q) a.dst[q * a.lp.plane + at] = out[q];
    } else {
#pragma unroll
        for (int q = 0; q < kQ; ++q) store_with_ghosts<1, kGhostP>(a.dst + q * a.lp.plane, a.lp, (int)i, (int)j, out[q]);
    }
}

// a = (u . grad) u by central differences of the ghosted u, k1 and k2 from D.
__global__ void pack_f64_kernel(double* pack, const double* uv, const double* Dh, PlaneLayout L, double magic,
                                double w2_fixed, int tau2_fixed) {
    const size_t n = (size_t)L.nx * L.ny, pl = L.plane;
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
        const int j = (int)(k / L.nx), i = (int)(k - (size_t)j * L.nx);
        const size_t o = L.at(i, j);
        const double *u = uv, *v = uv + pl;
        const double ux = u[o], uy = v[o];
        const double dxux = 0.5 * (u[o + 1] - u[o - 1]), dxuy = 0.5 * (v[o + 1] - v[o - 1]);
        const double dyux = 0.5 * (u[o + L.pitch] - u[o - L.pitch]), dyuy = 0.5 * (v[o + L.pitch] - v[o - L.pitch]);
        const double t1m = 3.0 * Dh[o];  // tau1 - 1/2 (Sec. 2.4); tau2 from Lambda (Eq. (28)) or fixed
        pack[o] = fma(ux, dxux, uy * dyux);
        pack[pl + o] = fma(ux, dxuy, uy * dyuy);
        pack[2 * pl + o] = 1.0 - 1.0 / (0.5 + t1m);
        pack[3 * pl + o] = 1.0 - (tau2_fixed ? w2_fixed : t1m / fma(0.5, t1m, magic));
    }
}

}  // namespace

cudaError_t launch_pack_f64(trtr_ctx* ctx) {
    const size_t n = (size_t)ctx->p.nx * ctx->p.ny, want = (n + 127) / 128, cap = (size_t)ctx->num_sms * 16;
    ctx->launches += 1;
    ctx->tables_new = true;
    const bool fixed = ctx->p.tau2_mode == TRTR_TAU2_FIXED;
    pack_f64_kernel<<<(unsigned)(want < cap ? want : cap), 128, 0, ctx->stream>>>(
        static_cast<double*>(ctx->pack64), static_cast<const double*>(ctx->uv), static_cast<const double*>(ctx->Dh),
        ctx->lf, ctx->p.magic, fixed ? 1.0 / ctx->p.tau2 : 0.0, fixed);
    return cudaGetLastError();
}

// One step from buffer `src` into dst as step `step`.  Blocks of one warp while they leave no SM with
// more than 16 of them, of four warps above.
cudaError_t launch_step_f64(trtr_ctx* ctx, const void* src, void* dst, long step) {
    if (!ctx->pack64_ready) {
        const cudaError_t e = launch_pack_f64(ctx);
        if (e != cudaSuccess) return e;
        ctx->pack64_ready = true;
    }
    // the tables and packed planes are read before the wait for the kernels before this one: the first
    // launch after their writer starts when that has completed
    const bool overlap = !ctx->tables_new;
    ctx->tables_new = false;
    F64Args a;
    a.src = static_cast<const double*>(src);
    a.dst = static_cast<double*>(dst);
    a.uv = static_cast<const double*>(ctx->uv);
    a.pack = static_cast<const double*>(ctx->pack64);
    const int cur = ctx->S_cur < 0 ? 0 : ctx->S_cur, prev = ctx->S_prev >= 0 ? ctx->S_prev : cur;
    a.s_n = static_cast<const double*>(ctx->S) + (ctx->S ? (size_t)cur * ctx->lf.plane : 0);
    a.s_p = static_cast<const double*>(ctx->S) + (ctx->S ? (size_t)prev * ctx->lf.plane : 0);
    a.pt = PulseTab::make(ctx->p.nx, ctx->p.ny);
    a.pulse = ctx->p.src_mode == TRTR_SRC_PULSE ? pulse_level<double>(ctx, a.pt, step) : nullptr;
    a.lp = ctx->lp;
    a.lf = ctx->lf;
    const unsigned n = (unsigned)ctx->p.nx * (unsigned)ctx->p.ny;
    const unsigned threads = n <= 32u * 16u * (unsigned)ctx->num_sms ? 32 : 128;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((n + threads - 1) / threads);
    cfg.blockDim = dim3(threads);
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = overlap;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    switch (ctx->p.src_mode) {
        case TRTR_SRC_FIELD: return cudaLaunchKernelEx(&cfg, f64_step_kernel<TRTR_SRC_FIELD>, a);
        case TRTR_SRC_PULSE: return cudaLaunchKernelEx(&cfg, f64_step_kernel<TRTR_SRC_PULSE>, a);
        default: return cudaLaunchKernelEx(&cfg, f64_step_kernel<TRTR_SRC_NONE>, a);
    }
}

TRTR_BOUNDS_TAKE(f64)

}  // namespace trtr
