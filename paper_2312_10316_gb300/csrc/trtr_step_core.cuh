// trtr_step_core.cuh -- device machinery of the fused TRT-R step shared by the single-grid
// kernel (trtr_step.cu) and the batched kernel (trtr_batch.cu): TMA / mbarrier helpers,
// packed FP32 pair arithmetic, the moment-space node update of Eq. (14), and the routines
// that compute one tile row from a shared-memory stage.  Tile geometry is BX x BY nodes
// (one warp per tile row).  Internal to the library.
#pragma once

#include <cudaTypedefs.h>

#include <string.h>

#include <type_traits>

#include "trtr_internal.cuh"

namespace trtr {
namespace core {

constexpr long long kWaitCycles = 4000000000LL;  // ~2 s at 2 GHz

template <typename S, int SRC, int BX, int BY>
struct Tile {
    using C = typename Store<S>::C;
    static constexpr int A = 16 / (int)sizeof(S);    // TMA x quantum of the populations
    static constexpr int PW = BX + A;                // population tile width
    static constexpr int AC = 16 / (int)sizeof(C);   // TMA x quantum of the fields
    static constexpr int UW = BX + 2 * AC;           // u tile width (halo rounded to AC)
    static constexpr int UH = BY + 2;
    static constexpr uint32_t pad128(uint32_t b) { return (b + 127) / 128 * 128; }
    // shared-memory tiles start on 128-byte boundaries (TMA destinations)
    static constexpr uint32_t POP_PLANE = pad128(BY * PW * sizeof(S));
    static constexpr int PLANE_ELEMS = POP_PLANE / sizeof(S);
    static constexpr uint32_t POP = kQ * POP_PLANE;
    static constexpr uint32_t U = pad128(2 * UH * UW * sizeof(C));
    static constexpr uint32_t D = pad128(BY * BX * sizeof(C));
    static constexpr uint32_t S_TILE = pad128(BY * BX * sizeof(C));
    static constexpr uint32_t SRCB = SRC == TRTR_SRC_FIELD ? 2 * S_TILE : 0;
    // bytes the TMA delivers per stage (the boxes, without the padding)
    static constexpr uint32_t TX = kQ * BY * PW * sizeof(S) + 2 * UH * UW * sizeof(C) + BY * BX * sizeof(C) +
                                   (SRC == TRTR_SRC_FIELD ? 2 * BY * BX * sizeof(C) : 0);
    static constexpr uint32_t STAGE = POP + U + D + SRCB;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return done != 0;
}

// Waits for the phase `parity` of `bar` to complete, for at most `limit` SM clock cycles.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, long long limit = kWaitCycles) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > limit) return false;
    }
    return true;
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
        "[%2];" ::"r"(smem_addr(dst)),
        "l"(map), "r"(smem_addr(bar)), "r"(x), "r"(y)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, "
        "%5}], [%2];" ::"r"(smem_addr(dst)),
        "l"(map), "r"(smem_addr(bar)), "r"(x), "r"(y), "r"(z)
        : "memory");
}

// L2 eviction priorities (createpolicy): loads whose tiles neighbouring CTAs read again (the
// halo) can ask to stay, stores that nothing in the launch reads again to leave first.
__device__ __forceinline__ uint64_t l2_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void tma_load_3d_hint(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z,
                                                 uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, "
        "{%3, %4, %5}], [%2], %6;" ::"r"(smem_addr(dst)),
        "l"(map), "r"(smem_addr(bar)), "r"(x), "r"(y), "r"(z), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void st_global_f2_hint(float* p, float2 v, uint64_t policy) {
    asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(p), "f"(v.x), "f"(v.y), "l"(policy)
                 : "memory");
}
// the same for a pair of 2-byte values (one 32-bit word)
template <typename S2>
__device__ __forceinline__ void st_global_b32_hint(S2* p, S2 v, uint64_t policy) {
    static_assert(sizeof(S2) == 4, "a 32-bit pair");
    uint32_t w;
    memcpy(&w, &v, sizeof(w));
    asm volatile("st.global.L2::cache_hint.b32 [%0], %1, %2;" ::"l"(p), "r"(w), "l"(policy) : "memory");
}

// Bulk copy of `bytes` (a multiple of 16) from shared to global memory, both addresses 16-byte
// aligned; the async proxy reads the source, completion is tracked per thread in bulk
// async-groups.
__device__ __forceinline__ void bulk_store(void* gdst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst), "r"(smem_addr(src)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// the shared-memory sources of this thread's bulk stores have been read (may be overwritten)
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// this thread's bulk stores are complete
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// generic-proxy writes to shared memory become visible to the async proxy (bulk stores)
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Checked builds (TRTR_BOUNDS_CHECK): a tiled TMA load's x coordinate times the element size is
// a multiple of 16 bytes and its shared-memory destination is 128-byte aligned; a load that
// breaks either is recorded and not issued (its barrier then times out, which is reported).
__device__ __forceinline__ bool tma_ok(const void* dst, int x, int y, int elem) {
#if TRTR_BOUNDS_CHECK
    if ((x * elem) % 16 != 0 || (smem_addr(dst) & 127u) != 0u) {
        TRTR_BOUNDS_FAULT(kBoundsTma, x, y);
        return false;
    }
#endif
    return true;
}

// Checked builds: a bulk copy of nb interior columns of row j from column i0 stays inside the
// interior row and has 16-byte aligned addresses and size; otherwise it is recorded and skipped.
template <typename S>
__device__ __forceinline__ bool bulk_ok(const S* gdst, const void* src, int i0, int j, int nb, const PlaneLayout& L) {
#if TRTR_BOUNDS_CHECK
    const unsigned bytes = (unsigned)nb * (unsigned)sizeof(S);
    if (i0 < 0 || i0 + nb > L.nx || j < 0 || j >= L.ny || (reinterpret_cast<uintptr_t>(gdst) & 15u) != 0u ||
        (smem_addr(src) & 15u) != 0u || (bytes & 15u) != 0u) {
        TRTR_BOUNDS_FAULT(kBoundsBulk, i0, j);
        return false;
    }
#endif
    return true;
}

// Entry of level n - 1 in the pulse tables for a batch launch of `steps` steps (the clock is advanced only
// after every CTA of the launch has finished its tiles); a clock outside the tables sets the flag.
__device__ __forceinline__ int table_entry_at(const BatchClock* clk, int steps, int* flag) {
    const volatile BatchClock* v = clk;
    BatchClock c = {};
    c.n = v->n;
    c.first = v->first;
    bool outside;
    const int e = c.table_entry(steps, &outside);
    if (outside && threadIdx.x == 0) atomicExch(flag, 1);
    return e;
}

// A CTA's end of a batch launch of `steps` steps (one thread), also of one whose wait gave up: the last CTA
// to finish advances the step clock and sets the work-list counter back.
__device__ __forceinline__ void advance_clock(BatchClock* clk, int steps) {
    __threadfence();
    if (atomicAdd(&clk->done, 1u) == gridDim.x - 1) {
        __threadfence();
        clk->n += steps;
        clk->next = 0;
        clk->done = 0;
        __threadfence();
    }
}

// Walks the linear tile indices t, t + stride, t + 2 stride, ... of a persistent CTA as
// (t mod m, t div m) without a division per tile: one division at the start, then an add and a
// carry per step (m: tiles per row of the order's rows).
struct TileCursor {
    int a, b, da, db, m;
    __device__ __forceinline__ void init(int t, int stride, int m_) {
        m = m_;
        a = t % m;
        b = t / m;
        da = stride % m;
        db = stride / m;
    }
    __device__ __forceinline__ void next() {
        a += da;
        b += db;
        if (a >= m) {
            a -= m;
            ++b;
        }
    }
};

// ---- arithmetic types --------------------------------------------------------------------
// FP32-computing storages work on pairs of adjacent nodes with the packed FP32 instructions
// of sm_100-family SMs (two lanes of FP32 per FADD2 / FMUL2 / FFMA2).
struct F2 {
    float2 v;
    __device__ __forceinline__ F2() {}
    __device__ __forceinline__ F2(float s) : v(make_float2(s, s)) {}
    __device__ __forceinline__ F2(float a, float b) : v(make_float2(a, b)) {}
    __device__ __forceinline__ explicit F2(float2 x) : v(x) {}
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return F2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return F2(__ffma2_rn(b.v, make_float2(-1.f, -1.f), a.v)); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return F2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) { return F2(__ffma2_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ F2 vdiv(F2 a, F2 b) { return F2(__fdividef(a.v.x, b.v.x), __fdividef(a.v.y, b.v.y)); }

// s = dt S^n + dt/2 (S^n - S^{n-1}) = 1.5 dt S^n - 0.5 dt S^{n-1} (a7, Eqs. (3) and (14)) of the
// manufactured source at the node pair (i, i + 1) (i even, images included) or the node i of row
// j, from the tables of the levels n - 1 and n (`lev`: level n - 1).
__device__ __forceinline__ F2 pulse_level_dt(F2 p1, F2 p2, float2 q) { return vfma(p1, F2(q.x), p2 * F2(q.y)); }
__device__ __forceinline__ F2 pulse_source_dt(const float* lev, const PulseTab& t, int i, int j) {
    if (!in_tables(t, i, 2, j)) return F2(0.f);
    auto level = [&](const float* p) {
        const float2 q = __ldg(reinterpret_cast<const float2*>(p + t.y + 2 * j));
        const F2 p1(__ldg(reinterpret_cast<const float2*>(p + i))), p2(__ldg(reinterpret_cast<const float2*>(p + t.p2 + i)));
        return pulse_level_dt(p1, p2, q);
    };
    return vfma(F2(1.5f), level(lev + t.level), F2(-0.5f) * level(lev));
}
__device__ __forceinline__ double pulse_source_dt(const double* lev, const PulseTab& t, int i, int j) {
    if (!in_tables(t, i, 1, j)) return 0.0;
    auto level = [&](const double* p) {
        const double2 q = __ldg(reinterpret_cast<const double2*>(p + t.y + 2 * j));
        return fma(__ldg(p + i), q.x, __ldg(p + t.p2 + i) * q.y);
    };
    return fma(1.5, level(lev + t.level), -0.5 * level(lev));
}

// The pulse tables of a tile of BX columns and BY rows in its stage: a box of LEVELS levels of P1 and P2 and, on
// the next 128-byte boundary, one of (Q1, Q2), loaded with the tile's populations.  Read from global
// memory by the lanes, the six loads a pair came behind the TMA loads of the tile and waited for L2, a level's
// entries being new to every launch (GB300, us a step, by the lanes / with the boxes; one step a launch: FP32 400^2
// 6.79 / 6.50, 16 x 8000 27.8 / 24.4, FP16 16 x 8000 20.6 / 18.1; two: FP32 400^2 4.75 / 4.57, 20000 x 32 9.50 / 8.88,
// FP16 2048^2 43.8 / 41.5).
template <int BX, int BY, int LEVELS>
struct TileTables {
    static constexpr int YOff = (LEVELS * 2 * BX * 4 + 127) / 128 * 128;
    static constexpr int TX = LEVELS * 2 * (BX + BY) * 4, Bytes = (YOff + LEVELS * 2 * BY * 4 + 127) / 128 * 128;
    static_assert(BX % 4 == 0 && BY % 2 == 0, "boxes on 16-byte boundaries");
    // columns from i0, rows from j0; entry: of the first level in the tables
    static __device__ __forceinline__ void issue(unsigned char* at, uint64_t* bar, const CUtensorMap* mx,
                                                 const CUtensorMap* my, int entry, int i0, int j0) {
        const int x = kTabGhost + i0, y = 2 * (kTabGhost + j0);
        if (tma_ok(at, x, entry, 4)) tma_load_3d(at, mx, bar, x, 0, entry);
        if (tma_ok(at + YOff, y, entry, 4)) tma_load_2d(at + YOff, my, bar, y, entry);
    }
    // the source term of the pair at column i0 + c, row j0 + r from the levels l and l + 1, as pulse_source_dt
    static __device__ __forceinline__ F2 source(const unsigned char* at, int l, int c, int r) {
        if (!in_tile(l, LEVELS - 1) || !in_tile(c, BX - 1) || !in_tile(r, BY)) return F2(0.f);
        auto level = [&](int k) {
            const float* x = reinterpret_cast<const float*>(at) + 2 * BX * k + c;
            const float* y = reinterpret_cast<const float*>(at + YOff) + 2 * BY * k + 2 * r;
            return pulse_level_dt(F2(*reinterpret_cast<const float2*>(x)), F2(*reinterpret_cast<const float2*>(x + BX)),
                                  *reinterpret_cast<const float2*>(y));
        };
        return vfma(F2(1.5f), level(l + 1), F2(-0.5f) * level(l));
    }
};

// The table fill.  FP64 takes r = x - c, z = r^2 / s^2 and exp(-z / 2) as they stand.  FP32 carries r, r^2, z and
// the exponent as unevaluated sums of two floats (exact products and sums: 45 bits and more), so that neither
// r near the pulse nor a large exponent costs digits, with no instruction of the FP64 pipe: in FP64, 14 of them an
// entry (16 cycles a warp each) made a fill of 20000 + 32 coordinates 39 us (GB300), now 12.5.
template <typename C>
struct PulseLevel;  // the pulse at one time level
template <>
struct PulseLevel<double> {
    double cx, cy, inv_s2, A;  // A: dt D0 D_amp s0^2 / s^4
    __host__ __device__ void set(const PulseTime& t, double amp) {
        cx = t.cx;
        cy = t.cy;
        inv_s2 = t.inv_s2;
        A = amp * t.amp * t.inv_s2;
    }
};
template <>
struct PulseLevel<float> {
    float2 cx, cy, inv_s2, e;  // (value, remainder); e: -log2(e) / (2 s^2)
    float A;
    static __host__ __device__ float2 split(double v) {
        float2 r;
        r.x = (float)v;
        r.y = (float)(v - (double)r.x);
        return r;
    }
    __host__ __device__ void set(const PulseTime& t, double amp) {
        cx = split(t.cx);
        cy = split(t.cy);
        inv_s2 = split(t.inv_s2);
        e = split(-0.5 * 1.4426950408889634074 * t.inv_s2);
        A = (float)(amp * t.amp * t.inv_s2);
    }
};

// (E sin, E [pi cos r + sin (1 - z)]) of coordinate w of the n along an axis at a level of centre c.
__device__ __forceinline__ double2 pulse_factors(const double* tab, int n, int w, double x0, double dx, double c,
                                                 const PulseLevel<double>& l) {
    const double sn = tab[w], cs = tab[n + w], r = x0 + w * dx - c, z = r * r * l.inv_s2, E = exp(-0.5 * z);
    return make_double2(E * sn, E * (3.14159265358979323846 * cs * r + sn * (1.0 - z)));
}
__device__ __forceinline__ float2 pulse_factors(const float* tab, int n, int w, double, double, float2 c,
                                                const PulseLevel<float>& l) {
    const float sn = tab[w], cs = tab[n + w], xh = tab[2 * n + w], xl = tab[3 * n + w];
    const float s = xh - c.x, b = s - xh;
    const float t = ((xh - (s - b)) - (c.x + b)) + (xl - c.y);
    const float rh = s + t, rl = t - (rh - s);  // r
    const float p = rh * rh, pe = fmaf(2.f * rh, rl, fmaf(rh, rh, -p));  // r^2
    const float a = p * l.e.x, ae = fmaf(p, l.e.x, -a) + fmaf(p, l.e.y, pe * l.e.x);
    const float k = rintf(a);
    const float E = k < -160.f ? 0.f : scalbnf(exp2f((a - k) + ae), (int)k);
    const float z = p * l.inv_s2.x, ze = fmaf(p, l.inv_s2.x, -z) + fmaf(p, l.inv_s2.y, pe * l.inv_s2.x);
    if (E == 0.f) return make_float2(0.f, 0.f);
    return make_float2(E * sn, E * (3.14159265358979323846f * cs * rh + sn * ((1.f - z) - ze)));
}

// Entry k of the tables, one coordinate of one level (levels[l]: of level l), coordinates outside the grid as
// their periodic images; `ready`: called before the stores.
constexpr unsigned table_entries(int nx, int ny) { return (unsigned)(nx + ny + 4 * kTabGhost) * kPulseLevels; }
template <typename C, class Ready>
__device__ __forceinline__ void fill_pulse_entry(const PulseFill& f, const PulseLevel<C>* levels, unsigned k, Ready&& ready) {
    const PulseTab t = PulseTab::make(f.nx, f.ny);
    const unsigned gx = f.nx + 2 * kTabGhost, per = gx + f.ny + 2 * kTabGhost;
    const unsigned lev = k / per, e = k - lev * per;
    const bool along_x = e < gx;
    const int n = along_x ? f.nx : f.ny, at = (int)(along_x ? e : e - gx) - kTabGhost;
    int w = at % n;
    w = w < 0 ? w + n : w;
    const PulseLevel<C>& l = levels[lev];
    const auto v = pulse_factors(static_cast<const C*>(along_x ? f.tab_x : f.tab_y), n, w, along_x ? f.x0 : f.y0, f.dx,
                                 along_x ? l.cx : l.cy, l);
    C* out = static_cast<C*>(f.tab) + kTabGhost + (size_t)lev * t.level;
    ready();
    if (!in_tables(t, along_x ? at : 0, 1, along_x ? 0 : at)) return;
    if (along_x) {
        out[at] = v.y;
        out[t.p2 + at] = v.x;
    } else {
        out[t.y + 2 * at] = l.A * v.x;
        out[t.y + 2 * at + 1] = l.A * v.y;
    }
}
// Entries k, k + stride, ...
template <typename C>
__device__ __forceinline__ void fill_pulse_tables(const PulseFill& f, const PulseLevel<C>* levels, unsigned k, unsigned stride) {
    for (const unsigned total = table_entries(f.nx, f.ny); k < total; k += stride) fill_pulse_entry(f, levels, k, [] {});
}

// The pulse at the time levels of one fill of the tables, computed on the host.
template <typename C>
struct PulseLevels {
    PulseLevel<C> t[kPulseLevels];
};
template <typename C>
inline PulseLevels<C> pulse_levels_of(const trtr_ctx* ctx, long first) {
    PulseLevels<C> l;
    const double amp = ctx->p.dt * ctx->pulse.D0 * ctx->pulse.D_amp;
    for (int k = 0; k < kPulseLevels; ++k) l.t[k].set(pulse_at(ctx->pulse, (double)(first + k) * ctx->p.dt), amp);
    return l;
}

inline PulseFill pulse_fill_of(const trtr_ctx* ctx) {
    PulseFill f;
    memset(static_cast<void*>(&f), 0, sizeof(f));
    f.tab = ctx->ptab;
    f.tab_x = ctx->tab_x;
    f.tab_y = ctx->tab_y;
    f.x0 = ctx->p.x0;
    f.y0 = ctx->p.y0;
    f.dx = ctx->p.dx;
    f.amp = ctx->p.dt * ctx->pulse.D0 * ctx->pulse.D_amp;
    f.nx = ctx->p.nx;
    f.ny = ctx->p.ny;
    return f;
}

// A fill of the context's tables with `pulse` from level `first` on has been launched (e: how that went).
inline void tables_filled(trtr_ctx* ctx, const Pulse& pulse, long first, cudaError_t e) {
    ctx->ptab_pulse = pulse;
    ctx->ptab_first = first;
    ctx->ptab_ready = e == cudaSuccess;
}

// The tables of a launch from step `step`: coordinate 0 of level step - 1.
template <typename C>
inline const C* pulse_level(const trtr_ctx* ctx, const PulseTab& t, long step) {
    return static_cast<const C*>(ctx->ptab) + kTabGhost + (size_t)(step - 1 - ctx->ptab_first) * t.level;
}

// The node update of Eq. (14) in moment space; g: pre-collision populations, out: P_i(x).
//
// OFS: g and out are the offsets h_i = g_i - w_i phi_ref of the 2-byte storages.  The offset
// folds into the moments: sum w_i = 1 gives phi = sum h_i + phi_ref; sum w_i e_i = 0 leaves the
// first moments alone; sum w_i (e_ia e_ib - d_ab/3) = 0 leaves B_ab alone when its trace part
// uses sum h_i / 3; and the rebuild is linear in m0 with weight w_i, so rebuilding from
// sum h_i + s (in place of phi + s) gives the offsets of the results.
template <typename V, bool OFS = false>
__device__ __forceinline__ void collide_node(const V g[kQ], V ux, V uy, V ax, V ay, V Dh, V s, V magic, V w2_fixed,
                                             bool tau2_fixed, V out[kQ], V phi_ref = V(0.f)) {
    using T = float;
    // relaxation rates: tau1 - 1/2 = 3 Dh (Sec. 2.4); tau2 from Lambda (Eq. (28)) or fixed
    const V t1m = V(T(3)) * Dh;
    const V w1 = vdiv(V(T(1)), V(T(0.5)) + t1m);
    const V w2 = tau2_fixed ? w2_fixed : vdiv(t1m, vfma(V(T(0.5)), t1m, magic));
    const V k1 = V(T(1)) - w1, k2 = V(T(1)) - w2;
    const V kh = vfma(V(T(-0.5)), w1, V(T(1)));

    // a2 + a4: moments (pair sums and differences of opposite directions)
    const V p12 = g[1] + g[2], p34 = g[3] + g[4], p56 = g[5] + g[6], p78 = g[7] + g[8];
    const V d12 = g[1] - g[2], d34 = g[3] - g[4], d56 = g[5] - g[6], d78 = g[7] - g[8];
    const V pdiag = p56 + p78;
    const V phis = (g[0] + p12) + (p34 + pdiag);  // sum of the inputs (phi, or phi - phi_ref)
    V phi = phis;
    if constexpr (OFS) phi = phis + phi_ref;
    const V jx = d12 + (d56 + d78);
    const V jy = d34 + (d56 - d78);
    const V pxx = p12 + pdiag;
    const V pyy = p34 + pdiag;
    const V pxy = p56 - p78;

    // a5 + a6 + a7: post-collision Hermite coefficients
    const V phux = phi * ux, phuy = phi * uy;
    const V euxx = phux * ux, euyy = phuy * uy, euxy = phux * uy;
    const V m0 = phis + s;  // (OFS: its rebuild gives offsets)
    const V m1x = vfma(kh, vfma(phi, ax, ux * s), vfma(k1, jx - phux, phux));
    const V m1y = vfma(kh, vfma(phi, ay, uy * s), vfma(k1, jy - phuy, phuy));
    const V third = phis * V(T(1.0 / 3.0));  // pairs with the input sums pxx, pyy
    const V Axx = vfma(k2, (pxx - third) - euxx, euxx);
    const V Ayy = vfma(k2, (pyy - third) - euyy, euyy);
    const V Axy = vfma(k2, pxy - euxy, euxy);
    const V Txxy = euxx * uy, Txyy = euxy * uy;

    // rebuild from even (E) and odd (O) halves of the opposite pairs, weights folded in:
    //   f_i = w_i [m0 + 3 e.m1 + 4.5 H2:A + 13.5 (H_xxy T_xxy + H_xyy T_xyy)]
    const V Asum = Axx + Ayy;
    const V m9 = m0 * V(T(1.0 / 9.0));
    const V E1 = vfma(V(T(-1.0 / 6.0)), Ayy, vfma(V(T(1.0 / 3.0)), Axx, m9));
    const V E3 = vfma(V(T(-1.0 / 6.0)), Axx, vfma(V(T(1.0 / 3.0)), Ayy, m9));
    const V O1 = vfma(V(T(-0.5)), Txyy, m1x * V(T(1.0 / 3.0)));
    const V O3 = vfma(V(T(-0.5)), Txxy, m1y * V(T(1.0 / 3.0)));
    const V Ed = vfma(V(T(1.0 / 12.0)), Asum, m0 * V(T(1.0 / 36.0)));
    const V E5 = vfma(V(T(0.25)), Axy, Ed);
    const V E7 = vfma(V(T(-0.25)), Axy, Ed);
    const V O5 = vfma(V(T(0.25)), Txxy + Txyy, (m1x + m1y) * V(T(1.0 / 12.0)));
    const V O7 = vfma(V(T(0.25)), Txyy - Txxy, (m1x - m1y) * V(T(1.0 / 12.0)));
    out[1] = E1 + O1;
    out[2] = E1 - O1;
    out[3] = E3 + O3;
    out[4] = E3 - O3;
    out[5] = E5 + O5;
    out[6] = E5 - O5;
    out[7] = E7 + O7;
    out[8] = E7 - O7;
    if constexpr (OFS) {
        out[0] = vfma(V(T(-2.0 / 3.0)), Asum, m0 * V(T(4.0 / 9.0)));
    } else {
        // The nine rebuilt values sum to m0 (the collision keeps phi + s, Sec. 2.2); the other
        // eight are the pairs E +- O, so the rest population is m0 - 2 (E1 + E3 + E5 + E7), which
        // equals w_0 m0 - (2/3)(A_xx + A_yy).  Formed the latter way the sum drifts: the rounded
        // weights 4/9, 1/9, 1/36 add up to 1 + 7.5e-9 in FP32, which multiplied the mass by that
        // every step.  Subtracting the four terms from m0 one at a time leaves a drift of a few
        // 1e-11 per step (summing the eight stored values first: 3e-10).
        out[0] = vfma(V(T(-2)), E1, vfma(V(T(-2)), E3, vfma(V(T(-2)), E5, vfma(V(T(-2)), E7, m0))));
    }
}

template <typename C>
__device__ __forceinline__ C weight(int q) {
    return q == 0 ? C(4.0 / 9.0) : (q < 5 ? C(1.0 / 9.0) : C(1.0 / 36.0));
}

// Columns of a tile row (of `valid` interior columns, at most 128) that one bulk copy writes: a
// whole number of 16-byte chunks.
template <typename S>
__device__ __forceinline__ int bulk_cols(int valid) {
    constexpr int kChunk = 16 / (int)sizeof(S);
    const int v = valid < 128 ? valid : 128;
    return v / kChunk * kChunk;
}

// Shared-memory column offset of plane q's tile (see the TMA origin in issue_tile).
template <int A>
__device__ __forceinline__ constexpr int plane_offset(int q) {
    return lattice_ex(q) == 1 ? A - 1 : (lattice_ex(q) == -1 ? 1 : 0);
}

// Pair (2-element) storage vectors and their conversion to / from packed FP32.
// Random bits of the stochastic rounding of node pair (i, i + 1) of row j (i even): the pair's
// key, and the 32 bits of its population q.
__device__ __forceinline__ uint32_t sr_pair_key(int i, int j, int nx, uint32_t rkey) {
    return sr_hash(((uint32_t)j * (uint32_t)nx + (uint32_t)i) ^ rkey);
}
#ifndef TRTR_SR_WORDS
#define TRTR_SR_WORDS 9
#endif
__device__ __forceinline__ uint32_t sr_bits(uint32_t rk, int q) {
    // 9 words (the key rotated by 7 q), or 3 or 1 words shared by groups of populations (sweeps)
    if (TRTR_SR_WORDS == 9) return __funnelshift_l(rk, rk, 7 * q);
    if (TRTR_SR_WORDS == 3) return q < 3 ? rk : (q < 6 ? rk * 0x85EBCA6Bu : rk * 0xC2B2AE35u);
    return rk;
}

// The bits of two nodes that are not one pair: each takes its half (h: 0 the first, 1 the second node of
// a pair) of its own pair's bits.
__device__ __forceinline__ uint32_t sr_mixed_bits(uint32_t ka, uint32_t kb, int ha, int hb, int q) {
    const uint32_t a = sr_bits(ka, q) >> (16 * ha), b = sr_bits(kb, q) >> (16 * hb);
    return (a & 0xffffu) | (b << 16);
}

template <typename S>
struct Pair;
template <>
struct Pair<float> {
    using type = float2;
    static __device__ __forceinline__ F2 decode(float2 v, float) { return F2(v); }
    static __device__ __forceinline__ F2 decode(float a, float b, float) { return F2(a, b); }
    static __device__ __forceinline__ float2 encode(F2 v, float) { return v.v; }
    static __device__ __forceinline__ F2 raw(float2 v) { return F2(v); }
    static __device__ __forceinline__ F2 raw(float a, float b) { return F2(a, b); }
    static __device__ __forceinline__ float2 encode_raw(F2 v) { return v.v; }
    static __device__ __forceinline__ float2 encode_sr(F2 v, uint32_t) { return v.v; }
};
template <>
struct Pair<__half> {
    using type = __half2;
    static __device__ __forceinline__ F2 decode(__half2 v, float off) {
        const float2 f = __half22float2(v);
        return F2(f.x + off, f.y + off);
    }
    static __device__ __forceinline__ F2 decode(__half a, __half b, float off) {
        return F2(__half2float(a) + off, __half2float(b) + off);
    }
    static __device__ __forceinline__ __half2 encode(F2 v, float off) {
        return __floats2half2_rn(v.v.x - off, v.v.y - off);
    }
    // the stored offsets themselves (their w_i phi_ref is folded into the moments)
    static __device__ __forceinline__ F2 raw(__half2 v) { return F2(__half22float2(v)); }
    static __device__ __forceinline__ F2 raw(__half a, __half b) { return F2(__half2float(a), __half2float(b)); }
    static __device__ __forceinline__ __half2 encode_raw(F2 v) { return __floats2half2_rn(v.v.x, v.v.y); }
    // stochastic rounding of both offsets, 32 random bits (the first node in the low half)
    static __device__ __forceinline__ __half2 encode_sr(F2 v, uint32_t rbits) {
        uint32_t d;
        asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(v.v.y), "f"(v.v.x), "r"(rbits));
        __half2 h;
        memcpy(&h, &d, sizeof(h));
        return h;
    }
};
template <>
struct Pair<__nv_bfloat16> {
    using type = __nv_bfloat162;
    static __device__ __forceinline__ F2 decode(__nv_bfloat162 v, float off) {
        const float2 f = __bfloat1622float2(v);
        return F2(f.x + off, f.y + off);
    }
    static __device__ __forceinline__ F2 decode(__nv_bfloat16 a, __nv_bfloat16 b, float off) {
        return F2(__bfloat162float(a) + off, __bfloat162float(b) + off);
    }
    static __device__ __forceinline__ __nv_bfloat162 encode(F2 v, float off) {
        return __floats2bfloat162_rn(v.v.x - off, v.v.y - off);
    }
    static __device__ __forceinline__ F2 raw(__nv_bfloat162 v) { return F2(__bfloat1622float2(v)); }
    static __device__ __forceinline__ F2 raw(__nv_bfloat16 a, __nv_bfloat16 b) {
        return F2(__bfloat162float(a), __bfloat162float(b));
    }
    static __device__ __forceinline__ __nv_bfloat162 encode_raw(F2 v) { return __floats2bfloat162_rn(v.v.x, v.v.y); }
    static __device__ __forceinline__ __nv_bfloat162 encode_sr(F2 v, uint32_t rbits) {
        uint32_t d;
        asm("cvt.rs.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(v.v.y), "f"(v.v.x), "r"(rbits));
        __nv_bfloat162 h;
        memcpy(&h, &d, sizeof(h));
        return h;
    }
};

template <typename S, int SRC, int BX, int BY>
__device__ __forceinline__ void issue_tile(unsigned char* stage, uint64_t* bar, const CUtensorMap* mp,
                                           const CUtensorMap* mu, const CUtensorMap* md, const CUtensorMap* ms,
                                           int i0, int j0, const StepArgs<typename Store<S>::C>& a, uint32_t more = 0) {
    using T = Tile<S, SRC, BX, BY>;
    mbar_expect_tx(bar, T::TX + more);
    constexpr int kPe = (int)sizeof(S), kFe = (int)sizeof(typename Store<S>::C);
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        const int x = i0 + a.lp.gx - (lattice_ex(q) == 1 ? T::A : 0);
        const int y = j0 + kGhostP - lattice_ey(q);
        if (tma_ok(stage + q * T::POP_PLANE, x, y, kPe)) tma_load_3d(stage + q * T::POP_PLANE, mp, bar, x, y, q);
    }
    const int yf = j0 + kGhostF;  // field row of the tile's first row
    if (tma_ok(stage + T::POP, i0 + a.lf.gx - T::AC, yf - 1, kFe))
        tma_load_3d(stage + T::POP, mu, bar, i0 + a.lf.gx - T::AC, yf - 1, 0);
    if (tma_ok(stage + T::POP + T::U, i0 + a.lf.gx, yf, kFe))
        tma_load_2d(stage + T::POP + T::U, md, bar, i0 + a.lf.gx, yf);
    if (SRC == TRTR_SRC_FIELD) {
        unsigned char* s = stage + T::POP + T::U + T::D;
        if (tma_ok(s, i0 + a.lf.gx, yf, kFe)) tma_load_3d(s, ms, bar, i0 + a.lf.gx, yf, a.s_cur);
        if (tma_ok(s + T::S_TILE, i0 + a.lf.gx, yf, kFe))
            tma_load_3d(s + T::S_TILE, ms, bar, i0 + a.lf.gx, yf, a.s_prev);
    }
}

// One tile row r of the FP32-computing storages, or NM * 64 columns of it from column c0: lane
// handles the node pairs (i0 + c0 + 64 m + 2 lane, + 1), m = 0 .. NM - 1.
//
// Stores: TST = false writes every value to global memory from the lanes.  TST = true (one warp
// per whole row) writes the row's nine result rows into shared memory over the row's own input
// rows (only this warp reads them; the results of pair m cover columns 64 m .. 64 m + 63, which
// no later pair reads), and lane 0 then copies each plane's row to global memory with one bulk
// copy of the row's first `bulk_cols(nx - i0)` columns (16-byte multiples: the row starts are
// 16-byte aligned in both memories).  The lanes store the few columns past those, and the ghost
// copies of edge nodes, directly.
// psrc: the source terms of the lane's pairs (TRTR_SRC_PULSE).
// UNR: the unroll factor of the pair loop (1: one pair at a time; NM: all pairs interleaved).
// SR: the 2-byte storages round stochastically (TRTR_ROUND_STOCHASTIC), with the random bits of
// sr_hash keyed by the node pair and a.rkey.
template <typename S, int SRC, int BX, int BY, int NM = BX / 64, bool TST = false, int UNR = 1, bool SR = false>
__device__ __forceinline__ void tile_row_pairs(const unsigned char* st, int r, int lane, int i0, int j,
                                               const StepArgs<float>& a, const F2* psrc, int c0 = 0) {
    static_assert(!TST || NM == BX / 64, "bulk row stores need one warp per tile row");
    using T = Tile<S, SRC, BX, BY>;
    using P = Pair<S>;
    using S2 = typename P::type;
    const int nx = a.lp.nx, ny = a.lp.ny;
    const S* sp = reinterpret_cast<const S*>(st) + r * T::PW;
    const float* su = reinterpret_cast<const float*>(st + T::POP) + (r + 1) * T::UW + T::AC;
    const float* sv = su + T::UH * T::UW;
    const float* sd = reinterpret_cast<const float*>(st + T::POP + T::U) + r * BX;
    const float* ss = reinterpret_cast<const float*>(st + T::POP + T::U + T::D) + r * BX;
    const float phi_ref = a.phi_ref;
    constexpr bool kOfs = sizeof(S) == 2;  // offset storages: h_i = g_i - w_i phi_ref, folded into the moments
    S* dst = static_cast<S*>(a.dst);
    const size_t pl = a.lp.plane;
    const F2 magic(a.magic), w2f(a.omega2_fixed);
#pragma unroll (UNR)
    for (int m = 0; m < NM; ++m) {
        const int c = c0 + 64 * m + 2 * lane;  // column of the pair inside the tile
        const int i = i0 + c;
        if (!TST && i >= nx) break;  // (TST: pairs past nx are computed; their columns are not stored)
        // a1: pull-streaming from the shifted tiles
        F2 g[kQ];
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const S* pq = sp + q * T::PLANE_ELEMS + c + plane_offset<T::A>(q);
            if (plane_offset<T::A>(q) % 2 == 0)
                g[q] = P::raw(*reinterpret_cast<const S2*>(pq));
            else
                g[q] = P::raw(pq[0], pq[1]);
        }
        // u, its central differences (ghosts make edges one-sided or periodic), D
        const float2 uc = *reinterpret_cast<const float2*>(su + c);
        const float2 vc = *reinterpret_cast<const float2*>(sv + c);
        const F2 ux(uc), uy(vc);
        const F2 dxux = F2(0.5f) * (F2(uc.y, su[c + 2]) - F2(su[c - 1], uc.x));
        const F2 dxuy = F2(0.5f) * (F2(vc.y, sv[c + 2]) - F2(sv[c - 1], vc.x));
        const F2 dyux = F2(0.5f) * (F2(*reinterpret_cast<const float2*>(su + c + T::UW)) -
                                    F2(*reinterpret_cast<const float2*>(su + c - T::UW)));
        const F2 dyuy = F2(0.5f) * (F2(*reinterpret_cast<const float2*>(sv + c + T::UW)) -
                                    F2(*reinterpret_cast<const float2*>(sv + c - T::UW)));
        const F2 ax = vfma(ux, dxux, uy * dyux);  // (u.grad) u_x
        const F2 ay = vfma(ux, dxuy, uy * dyuy);  // (u.grad) u_y
        const F2 Dh(*reinterpret_cast<const float2*>(sd + c));

        // a7: s = dt S^n + dt/2 (S^n - S^{n-1})
        F2 src(0.f);
        if (SRC == TRTR_SRC_FIELD) {
            const F2 sn(*reinterpret_cast<const float2*>(ss + c));
            const F2 sp_(*reinterpret_cast<const float2*>(ss + T::S_TILE / sizeof(float) + c));
            src = vfma(F2(1.5f), sn, F2(-0.5f) * sp_);
        } else if (SRC == TRTR_SRC_PULSE) {
            src = psrc[0];  // compile-time indices only (no local-memory array)
#pragma unroll
            for (int mm = 1; mm < NM; ++mm)
                if (m == mm) src = psrc[mm];
        }

        F2 out[kQ];
        // 2-byte storages: g and out stay offsets (the offset is folded into the moments)
        collide_node<F2, kOfs>(g, ux, uy, ax, ay, Dh, src, magic, w2f, a.tau2_fixed, out, F2(phi_ref));
        const uint32_t rk = SR ? sr_pair_key(i, j, nx, a.rkey) : 0u;
        auto enc = [&](int q) -> S2 {
            if constexpr (SR)
                return P::encode_sr(out[q], sr_bits(rk, q));
            else
                return P::encode_raw(out[q]);
        };

        // a8: store P_i(x); edge nodes also write their periodic ghost copies (the one-wide frame
        // that the one-step kernel reads)
        const bool edge = j == 0 || j == ny - 1 || i == 0 || i + 1 >= nx - 1;
        if constexpr (TST) {
            __syncwarp();  // every lane has read its inputs of pair m
            S* srow = const_cast<S*>(sp);
#pragma unroll
            for (int q = 0; q < kQ; ++q)
                *reinterpret_cast<S2*>(srow + q * T::PLANE_ELEMS + c) = enc(q);
            const int nb = bulk_cols<S>(nx - i0);
            if ((edge || c + 1 >= nb) && i < nx) {  // ghost copies, and the columns past the bulk copy
#pragma unroll
                for (int q = 0; q < kQ; ++q) {
                    const S2 v = enc(q);
                    const S v0 = reinterpret_cast<const S*>(&v)[0], v1 = reinterpret_cast<const S*>(&v)[1];
                    if (c >= nb) dst[q * pl + a.lp.at_g<kGhostP>(i, j)] = v0;
                    if (c + 1 >= nb && i + 1 < nx) dst[q * pl + a.lp.at_g<kGhostP>(i + 1, j)] = v1;
                    store_ghosts<1, kGhostP>(dst + q * pl, a.lp, i, j, v0);
                    if (i + 1 < nx) store_ghosts<1, kGhostP>(dst + q * pl, a.lp, i + 1, j, v1);
                }
            }
        } else if (!edge) {
            S* d0 = dst + a.lp.at_g<kGhostP>(i, j);
#if TRTR_BOUNDS_CHECK
            if (i + 1 >= nx || (reinterpret_cast<uintptr_t>(d0) % sizeof(S2)) != 0u) {
                TRTR_BOUNDS_FAULT(kBoundsPair, i, j);
                continue;
            }
#endif
#pragma unroll
            for (int q = 0; q < kQ; ++q)
                *reinterpret_cast<S2*>(d0 + q * pl) = enc(q);
        } else {
#pragma unroll
            for (int q = 0; q < kQ; ++q) {
                const S2 v = enc(q);
                store_with_ghosts<1, kGhostP>(dst + q * pl, a.lp, i, j, reinterpret_cast<const S*>(&v)[0]);
                if (i + 1 < nx) store_with_ghosts<1, kGhostP>(dst + q * pl, a.lp, i + 1, j, reinterpret_cast<const S*>(&v)[1]);
            }
        }
    }
    if constexpr (TST) {
        fence_proxy_async_smem();  // the result rows, for the bulk copies
        __syncwarp();
        const int nb = bulk_cols<S>(nx - i0);
        if (lane == 0 && nb > 0) {
#pragma unroll
            for (int q = 0; q < kQ; ++q)
                if (bulk_ok(dst + q * pl + a.lp.at_g<kGhostP>(i0, j), sp + q * T::PLANE_ELEMS, i0, j, nb, a.lp))
                    bulk_store(dst + q * pl + a.lp.at_g<kGhostP>(i0, j), sp + q * T::PLANE_ELEMS, (uint32_t)(nb * sizeof(S)));
            bulk_commit();
            bulk_wait_read();  // the stage may be refilled after the CTA barrier
        }
    }
}

// ---- host side: TMA descriptors --------------------------------------------------------

// L2 fill granularity of the TMA loads: 0 none, 1 64 B, 2 128 B, 3 256 B.
#ifndef TRTR_L2_PROMOTION
#define TRTR_L2_PROMOTION 0
#endif

template <typename S>
CUtensorMapDataType tma_type();
template <>
inline CUtensorMapDataType tma_type<float>() { return CU_TENSOR_MAP_DATA_TYPE_FLOAT32; }
template <>
inline CUtensorMapDataType tma_type<__half>() { return CU_TENSOR_MAP_DATA_TYPE_FLOAT16; }
template <>
inline CUtensorMapDataType tma_type<__nv_bfloat16>() { return CU_TENSOR_MAP_DATA_TYPE_BFLOAT16; }

inline PFN_cuTensorMapEncodeTiled_v12000 get_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

constexpr CUtensorMapL2promotion kPromotion =
    TRTR_L2_PROMOTION == 1   ? CU_TENSOR_MAP_L2_PROMOTION_L2_64B
    : TRTR_L2_PROMOTION == 2 ? CU_TENSOR_MAP_L2_PROMOTION_L2_128B
    : TRTR_L2_PROMOTION == 3 ? CU_TENSOR_MAP_L2_PROMOTION_L2_256B
                             : CU_TENSOR_MAP_L2_PROMOTION_NONE;

inline bool encode(CUtensorMap* m, CUtensorMapDataType t, int elem, void* base, const PlaneLayout& L, int depth, int bw,
            int bh, int bd) {
    auto fn = get_encoder();
    if (!fn) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)L.pitch, (cuuint64_t)L.rows, (cuuint64_t)depth};
    const cuuint64_t strides[2] = {(cuuint64_t)L.pitch * elem, (cuuint64_t)L.plane * elem};
    const cuuint32_t box[3] = {(cuuint32_t)bw, (cuuint32_t)bh, (cuuint32_t)bd};
    const cuuint32_t es[3] = {1, 1, 1};
    const cuuint32_t rank = depth > 1 ? 3 : 2;
    return fn(m, t, rank, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
              kPromotion, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The pulse tables as boxes of `levels` levels: `bx` columns of P1 and P2 (x), `by` rows of (Q1, Q2) (y).
inline bool encode_tables(CUtensorMap* x, CUtensorMap* y, void* tab, const PulseTab& t, int bx, int by, int levels) {
    auto fn = get_encoder();
    if (!fn) return false;
    const cuuint64_t xd[3] = {(cuuint64_t)t.p2, 2, (cuuint64_t)kPulseLevels};
    const cuuint64_t xs[2] = {(cuuint64_t)t.p2 * 4, (cuuint64_t)t.level * 4};
    const cuuint64_t yd[2] = {(cuuint64_t)(t.level - 2 * t.p2), (cuuint64_t)kPulseLevels};
    const cuuint64_t ys[1] = {(cuuint64_t)t.level * 4};
    const cuuint32_t xb[3] = {(cuuint32_t)bx, 2, (cuuint32_t)levels}, yb[2] = {(cuuint32_t)(2 * by), (cuuint32_t)levels};
    const cuuint32_t es[3] = {1, 1, 1};
    const auto f32 = CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    return fn(x, f32, 3, tab, xd, xs, xb, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, kPromotion,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS &&
           fn(y, f32, 2, static_cast<float*>(tab) + 2 * t.p2, yd, ys, yb, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, kPromotion, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// As encode, with bounds at the interior (coordinate 0 is node 0): loads outside it read zero, stores
// write nothing there.
inline bool encode_interior(CUtensorMap* m, CUtensorMapDataType t, int elem, void* base, const PlaneLayout& L, int depth,
                            int bw, int bh, int bd) {
    auto fn = get_encoder();
    if (!fn) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)L.nx, (cuuint64_t)L.ny, (cuuint64_t)depth};
    const cuuint64_t strides[2] = {(cuuint64_t)L.pitch * elem, (cuuint64_t)L.plane * elem};
    const cuuint32_t box[3] = {(cuuint32_t)bw, (cuuint32_t)bh, (cuuint32_t)bd};
    const cuuint32_t es[3] = {1, 1, 1};
    return fn(m, t, 3, static_cast<char*>(base) + ((size_t)L.gy * L.pitch + L.gx) * elem, dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, kPromotion,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace core
}  // namespace trtr
