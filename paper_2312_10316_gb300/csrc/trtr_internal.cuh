// trtr_internal.cuh -- context layout, storage traits and kernel launchers of the TRT-R
// library (not part of the public ABI).
//
// Device layout (all buffers owned by the context).  Every plane is "ghosted": the interior
// node (i, j) sits at row j + gy and column gx + i of a [rows][pitch] plane, where gx is one
// 128-byte line of columns, so interior rows start on a 128-byte boundary, and the gy columns
// before / after the interior and the gy rows above / below it hold ghost copies (gy = 2 for
// the populations, 1 for the fields of the one-step kernel, 4 for the packed fields; the sweep keeps
// four ghost columns of the populations):
//
//   populations  2 x [9][rows][pitch] in the storage type: the post-collision values P_i(x)
//                of the previous step; the pre-collision population is the pull
//                g_i(x, t_n) = P_i(x - e_i).  The ghost cells repeat the opposite edge
//                (periodic), so the pull never wraps and TMA tiles never need to.
//   fields       uv = [2][rows][pitch] (uhat_x, uhat_y) and Dh = [rows][pitch] in the compute
//                type, lattice units: uhat = u dt/dx, Dh = D dt/dx^2 (tau1 = 1/2 + 3 Dh).  The
//                u ghosts hold the periodic wrap (TRTR_GRAD_PERIODIC) or the linear
//                extrapolation 2u(edge) - u(edge -+ 1) (TRTR_GRAD_ONESIDED_EDGE), for which the
//                central difference at the edge node equals the one-sided difference.
//   source       [2][rows][pitch] dt*S in the compute type (TRTR_SRC_FIELD only)
//   packed       [5 or 6][rows][pitch] FP32: u, a = (u . grad) u, Dh and, with a source field, the
//                source term, for the kernels that take several steps; FP64: [4][rows][pitch]
//                a, k1, k2 (pack64)
//   pulse tab    [4][nx] sin(pi x_i), cos(pi x_i), x_i (two floats) and [4][ny] of y_j; and the
//                separable factors of the pulse source at kPulseLevels time levels (PulseTab)
//   edge values  [2 nx + 2 (ny - 2)] FP64 Dirichlet values of the edge nodes
//                (TRTR_BC_DIRICHLET_NEE), in the order of edge_node()
//   scratch      FP64 partial sums of the reductions, one pair per reduction block
//   flag         device int set by a kernel whose bounded wait gave up
// rows >= ny + 2 gy and pitch >= nx + 2 gx are padded so that every TMA box fits inside the
// allocation.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "trtr.h"

namespace trtr {

constexpr int kQ = 9;

struct Pulse {
    double omega, xc, yc, sigma0, D0, D_amp;
};
inline bool operator==(const Pulse& a, const Pulse& b) {
    return a.omega == b.omega && a.xc == b.xc && a.yc == b.yc && a.sigma0 == b.sigma0 && a.D0 == b.D0 && a.D_amp == b.D_amp;
}

// Per-time uniforms of the pulse source / closed form, computed on the host in double.
struct PulseTime {
    double cx, cy;    // centre c(t)
    double inv_s2;    // 1 / s^2(t)
    double amp;       // s0^2 / s^2(t)
};

// ---- bounds-checked builds (TRTR_BOUNDS_CHECK=1) ----------------------------------------
// The debug build checks the kernels' memory accesses against the layout: every plane index
// (PlaneLayout::at), where a kernel goes on from one index with offsets the outermost of them (in_frame), the
// pulse tables' entries (in_tables), the rows and columns of staged tiles and of the sweep's ring (in_tile), the
// pair stores, the bulk row copies and the TMA load coordinates.  An access out of bounds is recorded in this
// translation unit's log and then skipped, or kept inside the ghost frame; it never traps, so the context
// stays usable and the host reports TRTR_EBOUNDS at the next synchronisation.  The default build compiles
// none of it.  Not checked: the caller's [ny][nx] arrays and the library's own one-dimensional ones
// (reduction partials, edge values, work-lists), and TMA stores, which the hardware clips to the interior.
#ifndef TRTR_BOUNDS_CHECK
#define TRTR_BOUNDS_CHECK 0
#endif

enum BoundsKind {
    kBoundsPlane = 1,  // a plane index outside the interior and its ghost frame
    kBoundsPair = 2,   // a two-node store past the row or not aligned to the pair
    kBoundsBulk = 3,   // a bulk row copy outside the interior row, or not 16-byte aligned
    kBoundsTma = 4,    // a TMA load whose x coordinate or destination breaks the alignment rules
    kBoundsTile = 5,   // a column or row outside a staged tile or the sweep's ring (value, count)
    kBoundsTable = 6,  // an entry outside the pulse tables
};

#if TRTR_BOUNDS_CHECK
// [0] number of accesses caught, [1] kind of the first, [2] its (j << 32 | i); one log per
// translation unit (read and cleared by bounds_take_<unit>()).
static __device__ unsigned long long bounds_log[3];
__device__ __forceinline__ void bounds_fault(int kind, int i, int j) {
    if (atomicAdd(&bounds_log[0], 1ull) == 0ull) {
        bounds_log[1] = (unsigned long long)kind;
        bounds_log[2] = ((unsigned long long)(unsigned)j << 32) | (unsigned)i;
    }
}
#define TRTR_BOUNDS_FAULT(kind, i, j) ::trtr::bounds_fault((kind), (i), (j))
#else
#define TRTR_BOUNDS_FAULT(kind, i, j) ((void)0)
#endif

// Host side of a translation unit's log: copies {count, kind, where} to `out` and clears it
// (zeros in the default build).
#if TRTR_BOUNDS_CHECK
#define TRTR_BOUNDS_TAKE(unit)                                                                       \
    cudaError_t bounds_take_##unit(cudaStream_t s, unsigned long long* out) {                        \
        static const unsigned long long zero[3] = {0ull, 0ull, 0ull};                                \
        cudaError_t e = cudaMemcpyFromSymbolAsync(out, bounds_log, sizeof(zero), 0,                  \
                                                  cudaMemcpyDeviceToHost, s);                        \
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);                                          \
        if (e == cudaSuccess && out[0] != 0ull)                                                      \
            e = cudaMemcpyToSymbolAsync(bounds_log, zero, sizeof(zero), 0, cudaMemcpyHostToDevice, s); \
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);                                          \
        return e;                                                                                    \
    }
#else
#define TRTR_BOUNDS_TAKE(unit)                                                \
    cudaError_t bounds_take_##unit(cudaStream_t, unsigned long long* out) {   \
        out[0] = out[1] = out[2] = 0ull;                                      \
        return cudaSuccess;                                                   \
    }
#endif
cudaError_t bounds_take_step(cudaStream_t s, unsigned long long* out);
cudaError_t bounds_take_aux(cudaStream_t s, unsigned long long* out);
cudaError_t bounds_take_batch(cudaStream_t s, unsigned long long* out);
cudaError_t bounds_take_adjoint(cudaStream_t s, unsigned long long* out);
cudaError_t bounds_take_step2(cudaStream_t s, unsigned long long* out);
cudaError_t bounds_take_sweep(cudaStream_t s, unsigned long long* out);
cudaError_t bounds_take_f64(cudaStream_t s, unsigned long long* out);
cudaError_t bounds_take_small(cudaStream_t s, unsigned long long* out);
// All units: the summed count, and the kind and place of the first unit's first access.
cudaError_t bounds_take_all(cudaStream_t s, unsigned long long* out);

// Ghost frame widths: the population planes keep two ghost columns and rows on each side (the
// two-step kernel pulls twice across an edge); the field planes of the one-step kernel one.
constexpr int kGhostP = 2;
constexpr int kGhostF = 1;
constexpr int kGhostT = 4;  // the packed fields of the two- and four-step kernels

struct PlaneLayout {
    int nx, ny;
    int gx;        // column of interior x = 0 (128 bytes of columns)
    int gy;        // row of interior y = 0 = width of the ghost frame
    int pitch;     // elements per row
    int rows;      // rows per plane (>= ny + 2 gy)
    size_t plane;  // rows * pitch
    __host__ __device__ __forceinline__ size_t at(int i, int j) const { return at_w(i, j, gy); }
    // the same for a layout whose ghost width G is known at compile time (G == gy)
    template <int G>
    __host__ __device__ __forceinline__ size_t at_g(int i, int j) const {
        return at_w(i, j, G);
    }
    __host__ __device__ __forceinline__ size_t at_w(int i, int j, int g) const {
#if TRTR_BOUNDS_CHECK && defined(__CUDA_ARCH__)
        if (g != gy || i < -g || i >= nx + g || j < -g || j >= ny + g) {  // outside the interior and its ghost frame
            TRTR_BOUNDS_FAULT(kBoundsPlane, i, j);
            g = gy;
            i = i < -g ? -g : (i >= nx + g ? nx + g - 1 : i);
            j = j < -g ? -g : (j >= ny + g ? ny + g - 1 : j);
        }
#endif
        return (size_t)(j + g) * (size_t)pitch + (size_t)(i + gx);
    }
    // node (i, j) is in the interior or within wx columns and wy rows of it, and in the allocation
    __host__ __device__ bool covers(int i, int j, int wx, int wy) const {
        return i >= -wx && i < nx + wx && j >= -wy && j < ny + wy && i + gx >= 0 && i + gx < pitch && j + gy >= 0 && j + gy < rows;
    }
};
// Checked builds: false, and recorded, where an access is out of bounds, which the caller then skips.
__device__ __forceinline__ bool in_frame(const PlaneLayout& L, int i, int j, int wx, int wy) {
#if TRTR_BOUNDS_CHECK
    if (!L.covers(i, j, wx, wy)) {
        TRTR_BOUNDS_FAULT(kBoundsPlane, i, j);
        return false;
    }
#endif
    return true;
}
__device__ __forceinline__ bool in_tile(int v, int count) {
#if TRTR_BOUNDS_CHECK
    if (v < 0 || v >= count) {
        TRTR_BOUNDS_FAULT(kBoundsTile, v, count);
        return false;
    }
#endif
    return true;
}

PlaneLayout make_layout(int nx, int ny, int elem_bytes, int ghost);

// Storage traits: how a population is kept in memory and turned into the compute type.
template <typename S>
struct Store;

template <>
struct Store<double> {
    using C = double;
    static __device__ __forceinline__ double decode(double v, double) { return v; }
    static __device__ __forceinline__ double encode(double v, double) { return v; }
};

template <>
struct Store<float> {
    using C = float;
    static __device__ __forceinline__ float decode(float v, float) { return v; }
    static __device__ __forceinline__ float encode(float v, float) { return v; }
};

// Half-precision offset storage: h = g - w_i phi_ref.
template <>
struct Store<__half> {
    using C = float;
    static __device__ __forceinline__ float decode(__half v, float off) { return __half2float(v) + off; }
    static __device__ __forceinline__ __half encode(float v, float off) { return __float2half_rn(v - off); }
};

template <>
struct Store<__nv_bfloat16> {
    using C = float;
    static __device__ __forceinline__ float decode(__nv_bfloat16 v, float off) { return __bfloat162float(v) + off; }
    static __device__ __forceinline__ __nv_bfloat16 encode(float v, float off) { return __float2bfloat16_rn(v - off); }
};

// Tables of the pulse source (TRTR_SRC_PULSE).  With r = x - c(t) the manufactured source is a sum
// of two products of a function of x and a function of y,
//   dt S(x, y, t) = P1(x) Q1(y) + P2(x) Q2(y),
//   P2 = E(r_x) sin(pi x),  P1 = E(r_x) [pi cos(pi x) r_x + sin(pi x) (1 - r_x^2 / s^2)],
//   Q1 = A E(r_y) sin(pi y),  Q2 = A E(r_y) [pi cos(pi y) r_y + sin(pi y) (1 - r_y^2 / s^2)],
//   E(r) = exp(-r^2 / (2 s^2)),  A = dt D0 D_amp s0^2 / s^4,
// so a node's source costs four loads and two multiply-adds a time level instead of an exponential
// and a dozen operations; the tables of kPulseLevels time levels are filled by one small launch
// (nx + ny entries a level) when trtr_step leaves the levels they hold.  One level is
// [P1 over x][P2 over x][(Q1, Q2) over y], each with kTabGhost periodic images before and after
// the interior (halo nodes read their image's value without wrapping an index) and kTabPad unused
// entries behind them (ragged tiles).
constexpr int kPulseLevels = 64;
constexpr int kTabGhost = 8, kTabPad = 144;
struct PulseTab {
    int p2, y, level;  // offsets: P2 from P1, the y part from P1 (both at coordinate 0); stride of a level
    __host__ __device__ static PulseTab make(int nx, int ny) {
        const int wx = (kTabGhost + nx + kTabPad + 3) / 4 * 4, wy = (kTabGhost + ny + kTabPad + 3) / 4 * 4;
        PulseTab t;
        t.p2 = wx;
        t.y = 2 * wx + kTabGhost;  // kTabGhost values to P1's coordinate 0, 2 kTabGhost to (Q1, Q2)'s
        t.level = 2 * wx + 2 * wy;
        return t;
    }
    size_t values(int levels) const { return (size_t)level * levels; }
    // the entries of the columns [i, i + w) and of row j are in a level
    __host__ __device__ bool covers(int i, int w, int j) const {
        return i >= -kTabGhost && i + w <= p2 - kTabGhost && j >= -kTabGhost && j < (level - 2 * p2) / 2 - kTabGhost;
    }
};
__device__ __forceinline__ bool in_tables(const PulseTab& t, int i, int w, int j) {
#if TRTR_BOUNDS_CHECK
    if (!t.covers(i, w, j)) {
        TRTR_BOUNDS_FAULT(kBoundsTable, i, j);
        return false;
    }
#endif
    return true;
}

// Tile schedule bits of a step launch.  kSchedDynamic: the CTAs take their tiles from tile_ctr
// (long launches; kDynMinTilesPerCta).  kSchedReverse: the launch walks the tile order from the
// last tile to the first.  Consecutive launches on a context alternate the direction, so each
// starts on the tiles that the launch before it wrote last, whose lines are still in L2.
constexpr int kSchedDynamic = 1, kSchedReverse = 2;

// Uniform arguments of the fused step kernel (one launch per time step), a whole number of
// 16-byte chunks, so the batched kernel can copy them into shared memory with asynchronous
// 16-byte copies.
template <typename C>
struct alignas(16) StepArgs {
    void* dst;              // P written by this step (plain stores, with ghosts)
    const C* pulse;         // pulse tables of a batch's instance: coordinate 0 of their first level
    int* flag;              // set when a bounded wait gives up
    unsigned* tile_ctr;     // [next tile, CTAs done] of kernels that hand out tiles dynamically (zero between launches)
    PlaneLayout lp;         // populations
    PlaneLayout lf;         // fields
    int s_cur, s_prev;      // source buffer indices (TRTR_SRC_FIELD)
    int tau2_fixed;
    C magic;                // Lambda
    C omega2_fixed;         // 1 / tau2 (TRTR_TAU2_FIXED)
    C phi_ref;
    PulseTab pt;            // their layout
    int entry;              // of level n - 1 in the pulse tables (TRTR_SRC_PULSE; a context's)
    uint32_t rkey;          // stochastic rounding of the 2-byte storages: the step's key (sr_step_key)
    int sched;              // kSchedDynamic | kSchedReverse (below)
};

// Random bits of the stochastic rounding (TRTR_ROUND_STOCHASTIC): Wellons' "lowbias32"
// integer hash (two multiply / xor-shift rounds, published with its measured avalanche bias).
// The step's key hashes the step number; a node pair's key hashes its first node's index with
// the step key, and population q of the pair takes that key rotated by 7 q bits.  The bits
// depend on nothing but (node, step, q), so a run is the same however its steps are launched.
__host__ __device__ __forceinline__ uint32_t sr_hash(uint32_t x) {
    x ^= x >> 16;
    x *= 0x7feb352dU;
    x ^= x >> 15;
    x *= 0x846ca68bU;
    x ^= x >> 16;
    return x;
}
__host__ __device__ __forceinline__ uint32_t sr_step_key(long step) {
    return sr_hash((uint32_t)step * 0x9E3779B9U + (uint32_t)((unsigned long long)step >> 32) + 0x632BE5ABU);
}

// Programmatic dependent launch of the one- and two-step kernels: only for launches of a few tiles per CTA,
// where the launch latency it hides is a large part of the step.  On long launches it costs time
// (measured on GB300 without events between the launches: the two-step kernel at 4096^2 0.360
// against 0.346 ms, at 8192^2 1.97 against 1.41 ms; the one-step FP16 kernel at 8192^2 0.634
// against 0.612 ms), and a launch that records an event after it does not overlap anyway.  The sweep, whose
// CTAs have a share of rows each, takes it on every launch (us a step without / with: FP32 512^2 3.75 / 3.00,
// 1024^2 8.28 / 7.67, 4096^2 90.6 / 89.8, 8192^2 338.5 / 337.6; FP16 pulse 8192^2 408.3 / 409.0), and so do the
// small-grid and FP64 kernels.
constexpr long kPdlMaxTilesPerCta = 8;
// Tiles handed out from a counter: only for launches of more than this many tiles per CTA.  On
// short launches the CTAs' few sequential atomic round trips cost more than the balancing gains
// (the 512^2 adjoint's forward steps: 11 -> 18 us per two-step launch).
constexpr long kDynMinTilesPerCta = 8;

// (kMapS: the source planes, or the x factors of the pulse tables, whose y factors are kMapY)
enum MapId { kMapPop0 = 0, kMapPop1 = 1, kMapU = 2, kMapD = 3, kMapS = 4, kMapY = 5, kNumMaps = 6 };

// Whether tables that hold kPulseLevels time levels from `first` on hold those of a launch of `steps` steps
// from step `step`: step - 1 .. step + steps - 1.
__host__ __device__ inline bool levels_within(long first, long step, int steps) {
    return step - 1 >= first && step + steps <= first + kPulseLevels;
}

// Device clock of a batch.  Every launch that the host has counted advances it, one whose wait gave up
// too: the host's step and the clock's never part, and the tables' levels that the host has filled are those
// that the launches look up.
struct BatchClock {
    long long n;        // step of the instances
    unsigned int done;  // CTAs of the running launch that have finished
    unsigned int next;  // next work-list entry of a dynamically scheduled launch
    long long first;    // time level of the pulse tables' first entry
    // Entry of level n - 1 for a launch of `steps` steps, which reads the entries up to steps behind it.  A
    // clock outside the tables (*outside) is answered by their nearest entry: no launch reads past them.
    __host__ __device__ int table_entry(int steps, bool* outside) const {
        const long long e = n - 1 - first, last = kPulseLevels - 1 - steps;
        *outside = e < 0 || e > last;
        return (int)(e < 0 ? 0 : (e > last ? last : e));
    }
};

// The four-step kernel over a batch: its descriptors and work-list (device), and the work-list's length
// (rows of its busiest CTA, ramps included, and rows of an iteration).
struct SweepBatch {
    void *d_desc = nullptr, *d_units = nullptr, *d_first = nullptr;  // (one allocation)
    int ctas = 0, iteration_rows = 1;
    long rows = 0;
};

// What the table fill needs of a context or of a batch's instance.
struct PulseFill {
    void* tab;                       // [kPulseLevels][level]
    const void *tab_x, *tab_y;       // of the axes (trtr_ctx::tab_x)
    double x0, y0, dx, amp;          // amp: dt D0 D_amp
    int nx, ny;
};

}  // namespace trtr

struct trtr_adjoint_state;  // checkpoints and adjoint buffers (trtr_adjoint.cu)

struct trtr_ctx {
    CUtensorMap maps[trtr::kNumMaps];  // TMA descriptors (64-byte aligned type)
    trtr_params p;
    cudaStream_t stream;
    int device;
    int num_sms;
    int esize;        // bytes per stored population
    int csize;        // bytes per compute value (fields)
    trtr::PlaneLayout lp;  // population planes
    trtr::PlaneLayout lf;  // field planes
    void* pop[2];
    int cur;          // index of the buffer holding P for the current step
    void* uv;         // [2][rows][pitch] uhat_x, uhat_y
    void* Dh;
    void* S;          // [2][rows][pitch] (TRTR_SRC_FIELD)
    int S_cur;        // buffer holding S^n (-1: none set)
    int S_prev;       // buffer holding S^{n-1} (-1: use S^n)
    void* tab_x;      // [4][nx] sin and cos of pi x in the compute type; FP32: x as the sum of two floats
    void* tab_y;
    void* ptab;       // [kPulseLevels] pulse tables (TRTR_SRC_PULSE), behind tab_y ...
    void* ptab_own;   // ... or in an allocation of their own (an instance without a source beside ones with it)
    // what they hold, whoever filled them last (the context or its batch), if ptab_ready
    trtr::Pulse ptab_pulse;
    long ptab_first;  // time level of the first entry
    bool ptab_ready;
    bool tables_new;  // the tables or packed fields were written since the last launch that reads them early
                      // (before it waits for the launch before it)
    double* scratch;  // reduction partials
    int red_blocks;
    double* hres;     // pinned host memory that kernels write: the reductions' two results; [3]: copy of the timeout flag
    unsigned* red_done;  // blocks of a reduction that have finished (zero between reductions)
    int* dflag;       // device timeout flag; dflag[2], dflag[3]: tile counters
    double* dtmp;     // device staging for double I/O
    size_t dtmp_len;  // in doubles
    double* phib;     // Dirichlet values of the edge nodes (TRTR_BC_DIRICHLET_NEE)
    bool fields_set, pulse_set, initialized, maps_ready, dirichlet_set;
    bool small_tiles;  // step kernel geometry for small grids (chosen by encode_maps)
    // two-step kernel (FP32 storage, periodic boundaries, no source or the pulse source)
    CUtensorMap maps2[5];   // populations (buffers 0, 1), packed fields and pulse tables (x, y), its tile boxes
    CUtensorMap maps4[5];   // four-step kernel: population rows (buffers 0, 1), interior stores (0, 1), field rows
    void* fld2;             // [5 or 6][rows][pitch] float: uhat_x, uhat_y, a_x, a_y, Dh (and the stationary
                            // source term, TRTR_SRC_FIELD), four-wide periodic ghosts
    trtr::PlaneLayout lt;   // layout of fld2
    bool src_ready;         // its source plane (TRTR_SRC_FIELD) holds the current S^n
    bool fld2_ready;        // fld2 holds the current fields
    int sweep_rows;         // rows of its segments
    bool sweep_sooner;      // its four steps end before those of two two-step launches
    bool ghost4_ready;      // its four-wide ghost columns are up to date (interior rows)
    bool ghost2_ready;      // the current population buffer's whole two-wide ghost frame is up to date
    void* pack64;           // FP64: [4][rows][pitch] a_x, a_y, k1, k2 (the layout of uv)
    bool pack64_ready;      // it holds the current fields
    bool capturing;         // trtr_step is being captured into a graph: no four-step launches
    bool captured;          // a call of it has been: replays may change the tables and ghost frames between calls
    int steps_per_launch;   // 2: trtr_step uses the two-step kernel where it applies; 1: never
    trtr::Pulse pulse;
    long step;
    long launches;
    unsigned sweeps;        // step launches so far: the parity sets their tile direction (kSchedReverse)
    trtr_adjoint_state* adj;  // recorded forward run (trtr_forward_record), or NULL
    char err[512];
};

namespace trtr {

// Launchers (defined in trtr_step.cu and trtr_aux.cu).  All enqueue on ctx->stream and
// return the cudaGetLastError() of the launch.
cudaError_t encode_maps(trtr_ctx* ctx);
cudaError_t launch_step(trtr_ctx* ctx);
// one step from an arbitrary population buffer src (its map from encode_pop_map) into dst, as step `step`
cudaError_t launch_step_from(trtr_ctx* ctx, const void* src, const CUtensorMap* src_map, void* dst, long step);
cudaError_t launch_step_f64(trtr_ctx* ctx, const void* src, void* dst, long step);  // FP64 (trtr_f64.cu)
cudaError_t encode_pop_map(trtr_ctx* ctx, void* buffer, CUtensorMap* out);
// The two-step kernel: whether it applies to the context, its maps (at creation), the packed
// fields (after each change of u or D), and one launch advancing the state by two steps.
bool two_step_applies(const trtr_ctx* ctx);
cudaError_t encode_maps2(trtr_ctx* ctx);
cudaError_t launch_pack_fields2(trtr_ctx* ctx);  // (and the pulse tables from the current step on)
cudaError_t launch_step2(trtr_ctx* ctx);
// the distance-2 ghost cells of the current population buffer (or of buffer P) from its
// interior (periodic)
cudaError_t launch_refresh_ghosts2(trtr_ctx* ctx);
cudaError_t launch_refresh_ghosts2_buffer(trtr_ctx* ctx, void* P);
// the two-step kernel from an arbitrary population buffer (its map from encode_pop_map2) into
// dst, as steps `step` and `step + 1`; dst1 (or null) receives the intermediate state
cudaError_t encode_pop_map2(trtr_ctx* ctx, void* buffer, CUtensorMap* out);
cudaError_t launch_step2_from(trtr_ctx* ctx, const CUtensorMap* src_map, void* dst, void* dst1, long step);
// The four-step kernel (trtr_sweep.cu): whether it applies to the context, its maps (at creation),
// one launch advancing the state by four steps, and the ghost columns that it reads.
bool sweep_applies(const trtr_ctx* ctx);
double sweep_us(int precision, int src, double iterations);     // estimate of a launch of so many iterations a CTA
double two_step_us(int precision, int src, int num_sms, int nx, int ny);  // of a two-step launch (trtr_step2.cu)
cudaError_t encode_maps4(trtr_ctx* ctx);
cudaError_t launch_sweep(trtr_ctx* ctx);
cudaError_t launch_ghost_columns(trtr_ctx* ctx);
// the same four steps on a small grid (trtr_small.cu; reads no ghost cells)
bool small_applies(const trtr_ctx* ctx);
cudaError_t launch_small(trtr_ctx* ctx);
cudaError_t launch_pack_source(trtr_ctx* ctx);  // the source term's plane of the packed fields, from S^n
// The next launch of a run that may advance `most` (>= 1) steps, of a call that takes `call` in all:
// four, two or one steps, with what the launch needs; advances the context's state.  *taken: the
// steps; *what: names the failing launch on an error.
cudaError_t launch_steps(trtr_ctx* ctx, long most, long call, int* taken, const char** what);
// before the first and after the last launch_steps of a call (captured or not)
void begin_steps(trtr_ctx* ctx);
void end_steps(trtr_ctx* ctx);
// the same over a batch's instances (all of sweep_applies): setup, the ghost columns of buffer `parity`,
// one launch of four steps from buffer `parity` (odd: an instance of odd width)
cudaError_t sweep_batch_setup(trtr_ctx* const* ctx, int count, cudaStream_t stream, SweepBatch* out);
void sweep_batch_free(SweepBatch* b);
cudaError_t sweep_batch_ghost_columns(const SweepBatch& b, int count, int esize, int parity, cudaStream_t stream);
cudaError_t sweep_batch_launch(const SweepBatch& b, BatchClock* clk, int* flag, int parity, int precision, int src, bool sr,
                               bool odd, cudaStream_t stream);
// one block whose bounded wait on a barrier that nothing completes gives up after `cycles`
cudaError_t launch_wait_timeout(trtr_ctx* ctx, long long cycles);
// one thread that gives the bounds checks four bad arguments and accesses nothing with them
cudaError_t launch_bounds_probe(trtr_ctx* ctx);
void free_adjoint(trtr_ctx* ctx);
cudaError_t launch_convert_fields(trtr_ctx* ctx, const double* ux, const double* uy, const double* D);
cudaError_t launch_pulse_fields(trtr_ctx* ctx);
// The same into another buffer of the packed fields' layout, and the FP64 step's packed planes.
cudaError_t launch_pack_fields2_into(trtr_ctx* ctx, void* dst);
cudaError_t launch_pack_f64(trtr_ctx* ctx);
// Pulse tables: makes sure that they hold the time levels step - 1 .. step + steps - 1 (a launch
// where they do not), and the pointer that a launch from step `step` reads.
cudaError_t ensure_pulse_levels(trtr_ctx* ctx, long step, int steps);
cudaError_t launch_convert_source(trtr_ctx* ctx, const double* S, int buffer);
cudaError_t launch_init_equilibrium(trtr_ctx* ctx, const double* phi0 /* device or NULL = pulse */);
cudaError_t launch_moments(trtr_ctx* ctx, double* phi_out_dev);
cudaError_t launch_reduce(trtr_ctx* ctx, int kind, const double* phi_ref_dev);
cudaError_t launch_get_populations(trtr_ctx* ctx, double* g_dev);
cudaError_t launch_set_populations(trtr_ctx* ctx, const double* g_dev);
cudaError_t launch_sample(trtr_ctx* ctx, const long* nodes_dev, int count, double* out_dev);
// TRTR_BC_DIRICHLET_NEE: edge values from a device [ny][nx] array, and the boundary pass over
// the population buffer P that a step has just written
cudaError_t launch_gather_edges(trtr_ctx* ctx, const double* phi_b_dev);
cudaError_t launch_dirichlet(trtr_ctx* ctx, void* P);

// kReduceBadField: the number of values of the device array `ref` (one per node) that are not
// finite and positive (the check of a device-resident D).
enum ReduceKind { kReduceMass = 0, kReducePulse = 1, kReduceField = 2, kReduceNonFinite = 3, kReduceBadField = 4 };

__host__ __device__ inline PulseTime pulse_at(const Pulse& p, double t) {
    PulseTime r;
    const double c = cos(p.omega * t), s = sin(p.omega * t);
    r.cx = p.xc * c - p.yc * s;
    r.cy = p.xc * s + p.yc * c;
    const double s2 = p.sigma0 * p.sigma0 + 2.0 * p.D0 * t;
    r.inv_s2 = 1.0 / s2;
    r.amp = p.sigma0 * p.sigma0 / s2;
    return r;
}

// Edge nodes of an nx x ny grid (nx, ny >= 3), k in [0, 2 nx + 2 (ny - 2)): the bottom row,
// the top row, then the left and right columns without their corners.
__host__ __device__ inline int edge_count(int nx, int ny) { return 2 * nx + 2 * (ny - 2); }
__host__ __device__ inline void edge_node(int k, int nx, int ny, int* i, int* j) {
    if (k < nx) { *i = k; *j = 0; }
    else if (k < 2 * nx) { *i = k - nx; *j = ny - 1; }
    else if (k < 2 * nx + ny - 2) { *i = 0; *j = 1 + (k - 2 * nx); }
    else { *i = nx - 1; *j = 1 + (k - 2 * nx - (ny - 2)); }
}

// D2Q9 in the library's order: 0:(0,0) 1:(1,0) 2:(-1,0) 3:(0,1) 4:(0,-1) 5:(1,1) 6:(-1,-1)
// 7:(1,-1) 8:(-1,1).
__host__ __device__ constexpr int lattice_ex(int q) { return q == 1 || q == 5 || q == 7 ? 1 : (q == 2 || q == 6 || q == 8 ? -1 : 0); }
__host__ __device__ constexpr int lattice_ey(int q) { return q == 3 || q == 5 || q == 8 ? 1 : (q == 4 || q == 6 || q == 7 ? -1 : 0); }

// Stores one population value at every ghost cell that repeats interior node (i, j): the
// periodic images within W of the edges (W = 0: the layout's whole frame, L.gy wide), placed
// by a layout whose ghost width is GY (GY = 0: L.gy, read at run time; the step kernels know
// it at compile time).  The one-step kernels write the W = 1 frame that they read; the
// two-step kernel writes and reads the whole W = 2 frame (refresh_ghosts2 completes a frame
// left by one-step launches).
template <int W = 0, int GY = 0, typename T>
__device__ __forceinline__ void store_ghosts(T* plane, const PlaneLayout& L, int i, int j, T v) {
    const int w = W > 0 ? W : L.gy, g = GY > 0 ? GY : L.gy;
    const bool xl = i < w, xr = i >= L.nx - w, yl = j < w, yr = j >= L.ny - w;
    if (!(xl || xr || yl || yr)) return;
    if (xl) plane[L.at_w(i + L.nx, j, g)] = v;
    if (xr) plane[L.at_w(i - L.nx, j, g)] = v;
    if (yl) plane[L.at_w(i, j + L.ny, g)] = v;
    if (yr) plane[L.at_w(i, j - L.ny, g)] = v;
    if (xl && yl) plane[L.at_w(i + L.nx, j + L.ny, g)] = v;
    if (xl && yr) plane[L.at_w(i + L.nx, j - L.ny, g)] = v;
    if (xr && yl) plane[L.at_w(i - L.nx, j + L.ny, g)] = v;
    if (xr && yr) plane[L.at_w(i - L.nx, j - L.ny, g)] = v;
}

// Stores one population value at interior node (i, j) and at its ghost cells.
template <int W = 0, int GY = 0, typename T>
__device__ __forceinline__ void store_with_ghosts(T* plane, const PlaneLayout& L, int i, int j, T v) {
    plane[L.at_w(i, j, GY > 0 ? GY : L.gy)] = v;
    store_ghosts<W, GY>(plane, L, i, j, v);
}

}  // namespace trtr
