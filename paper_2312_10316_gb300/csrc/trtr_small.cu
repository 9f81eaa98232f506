// trtr_small.cu -- four time steps of the evolution equation (14) per launch for small grids (FP32
// storage or FP16 / BF16 offset storage, periodic; no source, the pulse source or a stationary source
// field).  On a grid of up to 300 nodes a side a launch is latency: the sweep's ramp
// (trtr_sweep.cu) makes it 6 - 10 us for four steps whatever the size, the two-step kernel takes 5 - 6 us
// for two.  Here a CTA takes one small tile with its four-node halo (32 x 8: 40 x 16 nodes), one node pair a
// thread, and every thread keeps its pair through the four steps: the fields, the source terms and the
// rounding keys stay in registers and are loaded while the launch before still runs, and only the
// populations pass through shared memory, in place (the node at step s reads and writes the slots
// x - s e_q, which no other node touches in that step), with one barrier a step.  The halo is computed
// again by every tile (2.5 pairs for each it keeps): with a few CTAs an SM that is time the SM would
// have idled.  Same bits as one step per launch.
#include "trtr_step_core.cuh"

namespace trtr {
namespace {

using namespace core;

constexpr int kT = 4;
// A BX x BY tile with its halo: W x H nodes, one pair a thread (whole warps).
template <int BX_, int BY_>
struct SmallTile {
    static constexpr int BX = BX_, BY = BY_, W = BX + 2 * kT, H = BY + 2 * kT, Pairs = W / 2;
    static constexpr int Threads = (Pairs * H + 31) / 32 * 32;
};

struct SmallArgs {
    const void* src;
    void* dst;
    const float* fields;  // packed fields
    const float* pulse;   // tables of level n - 1
    PulseTab pt;
    PlaneLayout lp, lt;
    int tau2_fixed;
    float magic, omega2_fixed, phi_ref;
    uint32_t rkey[kT];
};

// Step LV of the thread's pair at tile position (r, c).
template <typename S, int LV, int SRC, bool SR, class G>
__device__ __forceinline__ void small_step(S* tile, int r, int c, const F2 f[5], F2 src, const SmallArgs& a, uint32_t ka,
                                           uint32_t kb, bool mixed, int ha, int hb, int i, int j) {
    using S2 = typename Pair<S>::type;
    constexpr bool kOfs = sizeof(S) == 2;
    constexpr int kW = G::W, kH = G::H;
    if (r < LV || r >= kH - LV || c + 1 < LV || c >= kW - LV) return;
    auto slot = [&](int q) { return tile + (q * kH + r - LV * lattice_ey(q)) * kW + c - LV * lattice_ex(q); };
    auto even = [](int q) { return LV % 2 == 0 || lattice_ex(q) == 0; };
    if (!in_tile(r - LV, kH) || !in_tile(r + LV, kH)) return;
    // (a pair at the rim of a step's nodes reaches a column into the row beside it; one node of it is not used)
    if (!in_tile(r * kW + c - LV + 1, kH * kW) || !in_tile(r * kW + c + LV, kH * kW)) return;
    F2 g[kQ], out[kQ];
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        const S* s = slot(q);
        g[q] = even(q) ? Pair<S>::raw(*reinterpret_cast<const S2*>(s)) : Pair<S>::raw(s[0], s[1]);
    }
    collide_node<F2, kOfs>(g, f[0], f[1], f[2], f[3], f[4], src, F2(a.magic), F2(a.omega2_fixed), a.tau2_fixed, out,
                           F2(a.phi_ref));
    S2 v[kQ];
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        if constexpr (SR) {
            uint32_t bits = sr_bits(ka, q);
            if (mixed) bits = sr_mixed_bits(ka, kb, ha, hb, q);
            v[q] = Pair<S>::encode_sr(out[q], bits);
        } else {
            v[q] = Pair<S>::encode_raw(out[q]);
        }
    }
    if constexpr (LV < kT) {
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            S* s = slot(q);
            if (even(q)) {
                *reinterpret_cast<S2*>(s) = v[q];
            } else {
                s[0] = reinterpret_cast<const S*>(&v[q])[0];
                s[1] = reinterpret_cast<const S*>(&v[q])[1];
            }
        }
    } else {
        const int nx = a.lp.nx, ny = a.lp.ny;
        if (i >= nx || j >= ny) return;
        S* dst = static_cast<S*>(a.dst);
        if (i >= kGhostP && i + 1 < nx - kGhostP && j >= kGhostP && j < ny - kGhostP) {
            S* d = dst + a.lp.at_g<kGhostP>(i, j);
#pragma unroll
            for (int q = 0; q < kQ; ++q) *reinterpret_cast<S2*>(d + q * a.lp.plane) = v[q];
        } else {
#pragma unroll
            for (int q = 0; q < kQ; ++q) {
                S* plane = dst + q * a.lp.plane;
                store_with_ghosts<kGhostP, kGhostP>(plane, a.lp, i, j, reinterpret_cast<const S*>(&v[q])[0]);
                if (i + 1 < nx)
                    store_with_ghosts<kGhostP, kGhostP>(plane, a.lp, i + 1, j, reinterpret_cast<const S*>(&v[q])[1]);
            }
        }
    }
}

template <typename S, int SRC, bool SR, class G>
__global__ void __launch_bounds__(G::Threads, 2) small_kernel(const __grid_constant__ SmallArgs a) {
    using S2 = typename Pair<S>::type;
    constexpr int kW = G::W, kH = G::H, kPairs = G::Pairs, kBX = G::BX, kBY = G::BY;
    __shared__ __align__(16) S tile[kQ * kH * kW];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int nx = a.lp.nx, ny = a.lp.ny, tiles_x = (nx + kBX - 1) / kBX;
    const int ty = blockIdx.x / tiles_x, tx = blockIdx.x - ty * tiles_x;
    const int r = threadIdx.x / kPairs, c = 2 * (threadIdx.x - r * kPairs);  // (r >= kH: no pair)
    // the pair's node; past the halo of the last tiles (not used) it stays on the last halo nodes
    const int i = tx * kBX - kT + c, j = ty * kBY - kT + r;
    const int x = min(i, (nx + kT - 1) & ~1), y = min(j, ny + kT - 1);
    F2 f[5], src[kT];
    const float* fp = a.fields + a.lt.at_g<kGhostT>(x, y);
#pragma unroll
    for (int m = 0; m < 5; ++m) f[m] = F2(__ldg(reinterpret_cast<const float2*>(fp + m * a.lt.plane)));
#pragma unroll
    for (int s = 0; s < kT; ++s) {
        src[s] = F2(0.f);
        if (SRC == TRTR_SRC_PULSE) src[s] = pulse_source_dt(a.pulse + s * a.pt.level, a.pt, x, y);
        if (SRC == TRTR_SRC_FIELD) src[s] = F2(__ldg(reinterpret_cast<const float2*>(fp + 5 * a.lt.plane)));
    }
    auto wrap = [](int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); };
    const int xa = wrap(x, nx), xb = wrap(x + 1, nx), yw = wrap(y, ny);
    // rounding keys: of the pair, or, where an odd width lets a halo pair fall between the one-step
    // kernel's pairs, of each node's
    uint32_t ka[kT], kb[kT];
    const bool mixed = SR && (xa % 2 != 0 || xb != xa + 1);
    if (SR) {
#pragma unroll
        for (int s = 0; s < kT; ++s) {
            ka[s] = sr_pair_key(xa & ~1, yw, nx, a.rkey[s]);
            kb[s] = mixed ? sr_pair_key(xb & ~1, yw, nx, a.rkey[s]) : 0u;
        }
    } else {
#pragma unroll
        for (int s = 0; s < kT; ++s) ka[s] = kb[s] = 0u;
    }
    const S* P = static_cast<const S*>(a.src);
    const size_t pa = a.lp.at_g<kGhostP>(xa, yw), pb = a.lp.at_g<kGhostP>(xb, yw);
    const bool wide = xa % 2 == 0 && xb == xa + 1;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    S2 v[kQ];
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        if (wide) {
            v[q] = *reinterpret_cast<const S2*>(P + q * a.lp.plane + pa);
        } else {
            reinterpret_cast<S*>(&v[q])[0] = P[q * a.lp.plane + pa];
            reinterpret_cast<S*>(&v[q])[1] = P[q * a.lp.plane + pb];
        }
    }
    if (r < kH)
#pragma unroll
        for (int q = 0; q < kQ; ++q) *reinterpret_cast<S2*>(tile + (q * kH + r) * kW + c) = v[q];
    const int ha = xa & 1, hb = xb & 1;
    __syncthreads();
    small_step<S, 1, SRC, SR, G>(tile, r, c, f, src[0], a, ka[0], kb[0], mixed, ha, hb, i, j);
    __syncthreads();
    small_step<S, 2, SRC, SR, G>(tile, r, c, f, src[1], a, ka[1], kb[1], mixed, ha, hb, i, j);
    __syncthreads();
    small_step<S, 3, SRC, SR, G>(tile, r, c, f, src[2], a, ka[2], kb[2], mixed, ha, hb, i, j);
    __syncthreads();
    small_step<S, 4, SRC, SR, G>(tile, r, c, f, src[3], a, ka[3], kb[3], mixed, ha, hb, i, j);
}

template <class G>
long small_tiles(const trtr_ctx* ctx) {
    return (long)((ctx->p.nx + G::BX - 1) / G::BX) * ((ctx->p.ny + G::BY - 1) / G::BY);
}
// 32 x 4 tiles up to two CTAs an SM, then 32 x 8 up to two (FP32 without the pulse) or three, then the sweep.
// Measured (GB300, us a step; 32 x 4 / 32 x 8 / sweep).  FP32 without a source: 64^2 1.14 / 1.28 / -, 192^2 1.47 /
// 1.73 / 1.56, 256^2 2.17 / 1.78 / 1.84, 272^2 - / 2.15 / 1.83, 384^2 - / 2.90 / 2.47; a source field: 288^2 - / 2.24 /
// 1.94; the pulse, whose sweep has one warp a row: 256^2 - / 1.97 / 2.42, 320^2 - / 2.60 / 2.73, 336^2 - / 2.95 / 2.72;
// FP16: 256^2 - / 1.77 / 2.52, 320^2 - / 2.39 / 2.55, 352^2 - / 2.75 / 2.56.  (16 x 8 and 16 x 4 tiles: 1.31 and 1.39
// at 64^2, 1.63 and 1.65 at 192^2.)
using SmallA = SmallTile<32, 4>;
using SmallB = SmallTile<32, 8>;
constexpr long kSmallACtas = 2, kSmallBCtas = 3, kSmallBCtasF32 = 2;

template <typename S, int SRC, bool SR, class G>
cudaError_t launch_small_typed(trtr_ctx* ctx) {
    SmallArgs a;
    memset(static_cast<void*>(&a), 0, sizeof(a));
    a.src = ctx->pop[ctx->cur];
    a.dst = ctx->pop[ctx->cur ^ 1];
    a.fields = static_cast<const float*>(ctx->fld2);
    a.pt = PulseTab::make(ctx->p.nx, ctx->p.ny);
    a.pulse = SRC == TRTR_SRC_PULSE ? pulse_level<float>(ctx, a.pt, ctx->step) : nullptr;
    a.lp = ctx->lp;
    a.lt = ctx->lt;
    a.tau2_fixed = ctx->p.tau2_mode == TRTR_TAU2_FIXED;
    a.magic = (float)ctx->p.magic;
    a.omega2_fixed = (float)(ctx->p.tau2_mode == TRTR_TAU2_FIXED ? 1.0 / ctx->p.tau2 : 0.0);
    a.phi_ref = (float)ctx->p.phi_ref;
    for (int s = 0; s < kT; ++s) a.rkey[s] = sr_step_key(ctx->step + s);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)small_tiles<G>(ctx));
    cfg.blockDim = dim3(G::Threads);
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    // the fields and tables are read before the wait for the launch before: the first launch after their
    // writer starts when that has completed
    attr[0].val.programmaticStreamSerializationAllowed = !ctx->tables_new;
    ctx->tables_new = false;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, small_kernel<S, SRC, SR, G>, a);
}

template <typename S, int SRC, bool SR>
cudaError_t launch_small_geom(trtr_ctx* ctx) {
    return small_tiles<SmallA>(ctx) <= kSmallACtas * ctx->num_sms ? launch_small_typed<S, SRC, SR, SmallA>(ctx)
                                                                  : launch_small_typed<S, SRC, SR, SmallB>(ctx);
}

template <typename S, bool SR>
cudaError_t launch_small_src(trtr_ctx* ctx) {
    switch (ctx->p.src_mode) {
        case TRTR_SRC_FIELD: return launch_small_geom<S, TRTR_SRC_FIELD, SR>(ctx);
        case TRTR_SRC_PULSE: return launch_small_geom<S, TRTR_SRC_PULSE, SR>(ctx);
        default: return launch_small_geom<S, TRTR_SRC_NONE, SR>(ctx);
    }
}

}  // namespace

// Instead of the sweep (sizes: SmallA).
bool small_applies(const trtr_ctx* ctx) {
    const long ctas = ctx->p.precision == TRTR_F32 && ctx->p.src_mode != TRTR_SRC_PULSE ? kSmallBCtasF32 : kSmallBCtas;
    return sweep_applies(ctx) && small_tiles<SmallB>(ctx) <= ctas * ctx->num_sms;
}

cudaError_t launch_small(trtr_ctx* ctx) {
    const bool sr = ctx->p.rounding == TRTR_ROUND_STOCHASTIC;
    switch (ctx->p.precision) {
        case TRTR_F32: return launch_small_src<float, false>(ctx);
        case TRTR_F16_OFS: return sr ? launch_small_src<__half, true>(ctx) : launch_small_src<__half, false>(ctx);
        case TRTR_BF16_OFS:
            return sr ? launch_small_src<__nv_bfloat16, true>(ctx) : launch_small_src<__nv_bfloat16, false>(ctx);
        default: return cudaErrorInvalidValue;
    }
}

TRTR_BOUNDS_TAKE(small)

}  // namespace trtr
