// trtr_sweep.cu -- four time steps of the evolution equation (14) per launch: each CTA sweeps a
// strip of columns from bottom to top and carries four time levels behind one another through
// shared memory (wavefront temporal blocking), for FP32 storage or FP16 / BF16 offset storage
// (FP32 arithmetic), periodic boundaries and no source, the manufactured pulse source or a
// stationary source field.  The node update is the one-step kernel's, roundings included, so the
// results have the same bits.
//
// Strip: X = 120 output columns from i0; every level computes the 128 columns [i0 - 4, i0 + 124)
// (two node pairs a lane, or two warps a row), of which level s is valid on all but s - 1 at each side.
// Rows arrive through TMA, one box of the nine populations (136 columns from i0 - 8) and one of
// the five or six packed fields (128 columns from i0 - 4) a row, into a ring of Ring rows; y wraps by
// the row index, x through a four-wide ghost frame of columns.  Populations live in place: node x at
// level s reads and writes the slots x - s e_q of the ring, which no other node touches at that
// level, so one ring serves every level (level s = 1 .. 4 of row j uses the slot rows j - s, j,
// j + s).  In iteration k level s works on R rows, Lag rows behind level s - 1, which has then
// finished the row above them; an mbarrier per level and iteration is all that orders the warps (one
// CTA barrier an iteration: 144 GLUPS against 155).  The last level writes its rows to a shared-memory
// buffer that one TMA store an iteration moves out, clipped to the grid's whole 16-byte chunks; its
// lanes store the edge columns' ghost copies and the last columns themselves.
//
// Work units are (strip, segment of rows); a segment costs C rows of ramp (its first output row
// needs C / R iterations), so the host picks the number of segments that ends soonest.
//
// What bounds it: latency and issue, not memory.  At 2048^2 FP32 without a source 0.58 instructions are
// issued a cycle and scheduler, the shared-memory data path is 59 % busy, and DRAM carries 0.38 GB of the
// 0.39 GB a launch has to move; the warps wait for the level before theirs (a third of their time) and on
// fixed latencies.  Four steps move the populations once (92 B a node instead of 4 x 84), and 128 columns
// keep the work done twice at 128 / 120 plus the ramp.  Measured (GB300), us a step, the two-step kernel
// before -> now: FP32 pulse 4096^2 147 -> 99, no source 128 -> 89, FP16 pulse 139 -> 108; 200 steps of the
// FP32 pulse at 1024^2 with their set-up 3.43 -> 1.94 ms.
#include <algorithm>
#include <queue>
#include <utility>
#include <vector>

#include "trtr_step_core.cuh"

namespace trtr {
namespace {

using namespace core;

constexpr int kT = 4;                 // time levels of a launch
constexpr int kX = 120, kWC = 128;    // output and computed columns of a strip
constexpr int kW = kWC + 2 * kT;      // staged population columns
// packed fields: u, a, D and, with a stationary source field, the source term
__host__ __device__ constexpr int fields_of(int src) { return src == TRTR_SRC_FIELD ? 6 : 5; }
constexpr int kGhostX = 4;            // ghost columns that the strips read

template <typename S, int SRC>
struct Sweep {
    static constexpr int ES = (int)sizeof(S), NF = fields_of(SRC);
    // rows of an iteration, blocks loaded ahead: FP32 has room for 3 rows with five fields a row, 2 with
    // the source's (4096^2 without a source: 3 rows 163 GLUPS, 2 rows 146); 2-byte storages 4 rows
    static constexpr int R = ES == 2 ? 4 : (SRC == TRTR_SRC_FIELD ? 2 : 3);
    static constexpr int Ahead = ES == 2 ? 3 : (SRC == TRTR_SRC_FIELD ? 2 : 1);
    static constexpr int Lag = R + 1;
    static constexpr int C = ((kT - 1) * (Lag + 1) + R - 1) / R * R;  // ramp rows of a segment
    static constexpr int Ring = ((kT - 1) * Lag + kT + 1 + (Ahead + 1) * R + R - 1) / R * R;
    static constexpr int Blocks = Ring / R;
    static constexpr int PopRow = kQ * kW * ES, FldRow = NF * kWC * 4;
    static constexpr int OutBytes = (kQ * R * kX * ES + 127) / 128 * 128;
    static constexpr int FldOff = Ring * ((PopRow + 127) / 128 * 128);
    static constexpr int PopPitch = (PopRow + 127) / 128 * 128;       // TMA destinations on 128 bytes
    static constexpr int OutOff = FldOff + Ring * FldRow;
    static constexpr int Outs = 3;                                    // output buffers (two measured the same)
    static constexpr int BarOff = OutOff + Outs * OutBytes;
    static constexpr int Depth = 8;                                   // barriers of a level (iterations in flight)
    static constexpr int Smem = BarOff + (Blocks + kT * Depth + Outs) * 8 + 128;
    // Node pairs of a lane.  One (two warps a row) hides more latency, two (one warp) spend fewer instructions
    // on addresses and waits.  4096^2 FP32, us a step, one / two: no source 89.4 / 95.5, source field
    // (2048^2) 29.9 / 36.3, pulse (whose row factors every warp loads) 105.8 / 98.9; 2-byte storages 103 (three
    // rows: four would be 33 warps) / 96.
    static constexpr int P = ES == 4 && SRC != TRTR_SRC_PULSE ? 1 : 2;
    // The fields and the pulse tables are older than the launch before and are read while it still runs: FP32, us a
    // step, 512^2 3.09 -> 2.99, 1024^2 7.83 -> 7.63; FP16 pulse 4096^2 108.2 -> 109.1, so 2-byte storages wait first.
    static constexpr bool Early = ES == 4;
    static constexpr int Row = 2 / P;                                 // warps of a row
    static constexpr int Warps = kT * R * Row;                        // warps of a level: R rows
    static constexpr int Threads = (Warps + 1) * 32;                  // and one warp that moves the data
    static_assert(FldRow % 128 == 0, "TMA destinations on 128 bytes");
    // level 4 may finish iteration k when level 2 has finished k - 2, and level 1 may then be in k + 1 + Ahead
    static_assert(Ahead + 2 <= Depth, "a level stays within Depth iterations of the next");
    static_assert(Smem <= 227 * 1024, "the rings must fit in shared memory");
};

struct SweepArgs {
    const float* pulse;  // tables of level n - 1
    PulseTab pt;
    void* dst;
    int* flag;
    PlaneLayout lp;
    int gxf, gyf;        // interior origin of the packed fields
    int strips, seg_rows, units;
    int tau2_fixed;
    float magic, omega2_fixed, phi_ref;
    uint32_t rkey[kT];
};

// A batch launch works on the strips of its instances: unit u = units[u] = (instance, i0, j0, j1), CTA b's from
// first[b] on; the step and its tables' levels come from the batch's clock.
struct alignas(64) SweepDesc {
    CUtensorMap mp[2], mo[2], mf;  // by buffer
    SweepArgs a[2];                // by source buffer; pulse: the tables' first level
    void* pop[2];
};
struct ManyGrids {
    const SweepDesc* desc;
    const int4* units;
    const int* first;
    BatchClock* clk;
    int* flag;
    int parity;
};

// Columns of an nx-wide row in whole 16-byte chunks.
template <typename T>
__host__ __device__ __forceinline__ int bulk_cols_of(int nx) {
    constexpr int kChunk = 16 / (int)sizeof(T);
    return nx / kChunk * kChunk;
}

// The copies of one value of interior node (i, j) in the kGhostP ghost rows, corners included.
template <typename T>
__device__ __forceinline__ void store_row_ghosts(T* plane, const PlaneLayout& L, int i, int j, T v) {
    const int xs = i < kGhostX ? L.nx : (i >= L.nx - kGhostX ? -L.nx : 0);
    const int ys = j < kGhostP ? L.ny : -L.ny;
    if (!in_frame(L, i, j + ys, 0, kGhostP) || !in_frame(L, i + xs, j + ys, kGhostX, kGhostP)) return;
    T* row = plane + (ptrdiff_t)(j + kGhostP + ys) * L.pitch + L.gx;
    row[i] = v;
    if (xs) row[i + xs] = v;
}

// How a sweep rounds 2-byte values: to nearest (or FP32, not at all); stochastically; stochastically on
// an odd width, where halo pairs fall between the one-step kernel's pairs and every pair takes the
// bits of its two nodes' own pairs (two keys and a byte permutation, 8 % more instructions).
enum SweepRounding { kRoundNearest = 0, kRoundPairs = 1, kRoundNodes = 2 };
struct RoundKey {
    uint32_t a, b, sel;  // the two nodes' keys; the permutation that takes each one's half
};

// Level LV of row j for one lane: its G::P node pairs, at the columns c = 64 part + 2 lane and, with two,
// c + 64 (h = 0, 1), computed side by side.  pm / p0 / pp: the ring rows of the
// slots j - LV, j, j + LV, f: the row's fields, src: the source terms, rk: the rounding keys, at
// the first pair.  LV < kT writes the slots back, LV = kT the output buffer (and the ghost copies of
// rows within kGhostP of an edge).
template <typename S, int LV, int SRC, int RND, class G, class Wait>
__device__ __forceinline__ void sweep_row(S* pm, S* p0, S* pp, const float* f, const F2 src[G::P], const SweepArgs& a,
                                          const RoundKey rk[G::P], S* out_row, int lane, int part, int i, int j,
                                          Wait&& buffer_free) {
    constexpr bool kOfs = sizeof(S) == 2;
    using S2 = typename Pair<S>::type;
    F2 out[G::P][kQ];
    auto slot = [&](int q, int h) -> S* {
        S* row = lattice_ey(q) == 1 ? pm : (lattice_ey(q) == -1 ? pp : p0);
        return row + q * kW - LV * lattice_ex(q) + 64 * h;
    };
    auto even = [](int q) { return LV % 2 == 0 || lattice_ex(q) == 0; };
    F2 g[G::P][kQ], fld[G::P][G::NF];
#pragma unroll
    for (int h = 0; h < G::P; ++h) {
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const S* s = slot(q, h);
            g[h][q] = even(q) ? Pair<S>::raw(*reinterpret_cast<const S2*>(s)) : Pair<S>::raw(s[0], s[1]);
        }
#pragma unroll
        for (int m = 0; m < G::NF; ++m) fld[h][m] = F2(*reinterpret_cast<const float2*>(f + m * kWC + 64 * h));
    }
#pragma unroll
    for (int h = 0; h < G::P; ++h)
        collide_node<F2, kOfs>(g[h], fld[h][0], fld[h][1], fld[h][2], fld[h][3], fld[h][4],
                               SRC == TRTR_SRC_FIELD ? fld[h][G::NF - 1] : src[h], F2(a.magic),
                               F2(a.omega2_fixed), a.tau2_fixed, out[h], F2(a.phi_ref));
    auto enc = [&](int q, int h) -> S2 {
        if constexpr (RND == kRoundPairs)
            return Pair<S>::encode_sr(out[h][q], sr_bits(rk[h].a, q));
        else if constexpr (RND == kRoundNodes)
            return Pair<S>::encode_sr(out[h][q], __byte_perm(sr_bits(rk[h].a, q), sr_bits(rk[h].b, q), rk[h].sel));
        else
            return Pair<S>::encode_raw(out[h][q]);
    };
    if constexpr (LV < kT) {
#pragma unroll
        for (int h = 0; h < G::P; ++h)
#pragma unroll
            for (int q = 0; q < kQ; ++q) {
                const S2 v = enc(q, h);
                S* s = slot(q, h);
                if (even(q)) {
                    *reinterpret_cast<S2*>(s) = v;
                } else {
                    s[0] = reinterpret_cast<const S*>(&v)[0];
                    s[1] = reinterpret_cast<const S*>(&v)[1];
                }
            }
    } else {
        if (!buffer_free()) return;  // (a wait gave up: the warp leaves at its next wait)
        const int nx = a.lp.nx, nc = bulk_cols_of<S>(nx);
#pragma unroll
        for (int h = 0; h < G::P; ++h) {
            if (part + h == 0 ? lane < kT / 2 : lane >= 32 - kT / 2) continue;  // outside the output columns
            if (!in_tile(2 * lane + 64 * (part + h) - kT, kX - 1)) continue;
            const int ih = i + 64 * h;
            S2 v[kQ];
#pragma unroll
            for (int q = 0; q < kQ; ++q) {
                v[q] = enc(q, h);
                *reinterpret_cast<S2*>(out_row + q * (G::R * kX) + 64 * h) = v[q];
            }
            // the edge columns from the registers (copied from the buffer by the data mover, the edge strips took
            // 2950 cycles an iteration, the others 2200: a 1024^2 step 10.1 us, now 8.6)
            if (ih < kGhostX || ih + 1 >= min(nx - kGhostX, nc)) {
                S* row = static_cast<S*>(a.dst) + (size_t)(j + kGhostP) * a.lp.pitch + a.lp.gx + ih;
                const int to = ih < kGhostX ? nx : -nx;
                const bool g0 = ih < kGhostX || (ih >= nx - kGhostX && ih < nx);
                const bool g1 = ih < kGhostX || (ih + 1 >= nx - kGhostX && ih + 1 < nx);
                const bool t0 = ih >= nc && ih < nx, t1 = ih + 1 >= nc && ih + 1 < nx;
#pragma unroll
                for (int q = 0; q < kQ; ++q) {
                    S* r = row + q * a.lp.plane;
                    const S v0 = reinterpret_cast<const S*>(&v[q])[0], v1 = reinterpret_cast<const S*>(&v[q])[1];
                    if (g0 && in_frame(a.lp, ih + to, j, kGhostX, 0)) r[to] = v0;
                    if (g1 && in_frame(a.lp, ih + to + 1, j, kGhostX, 0)) r[to + 1] = v1;
                    if (t0 && in_frame(a.lp, ih, j, 0, 0)) r[0] = v0;
                    if (t1 && in_frame(a.lp, ih + 1, j, 0, 0)) r[1] = v1;
                }
            }
            if (j < kGhostP || j >= a.lp.ny - kGhostP) {
#pragma unroll 1
                for (int q = 0; q < kQ; ++q) {
                    const S* v = out_row + q * (G::R * kX) + 64 * h;
                    S* plane = static_cast<S*>(a.dst) + q * a.lp.plane;
                    if (ih < nx) store_row_ghosts(plane, a.lp, ih, j, v[0]);
                    if (ih + 1 < nx) store_row_ghosts(plane, a.lp, ih + 1, j, v[1]);
                }
            }
        }
    }
}

__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, const void* src, int x, int y, int z) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(map),
                 "r"(smem_addr(src)), "r"(x), "r"(y), "r"(z)
                 : "memory");
}

__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// One context (BATCH = false): mp_ population rows of the source, mf_ field rows, mo_ interior of the result;
// unit u = (strip, segment), taken by the CTAs in turn.  BATCH: many alone.
template <typename S, int SRC, int RND, class G, bool BATCH>
__global__ void __launch_bounds__(G::Threads, 1)
    sweep_kernel(const __grid_constant__ CUtensorMap mp_, const __grid_constant__ CUtensorMap mf_,
                 const __grid_constant__ CUtensorMap mo_, const __grid_constant__ SweepArgs a_,
                 const __grid_constant__ ManyGrids p) {
    using Args = std::conditional_t<BATCH, SweepArgs, const SweepArgs&>;  // (batch: copied once a unit)
    constexpr int R = G::R;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int s_abort;
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) &
                                                           ~static_cast<uintptr_t>(127));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + G::BarOff);  // [Blocks]: a block of rows has arrived
    uint64_t* done = full + G::Blocks;                               // [kT][Depth]: a level has finished an iteration
    uint64_t* freed = done + kT * G::Depth;                          // [Outs]: an output buffer has been stored
    const int tid = threadIdx.x, lane = tid & 31, w = __shfl_sync(0xffffffffu, tid >> 5, 0);
    if (tid == 0) {
        s_abort = 0;
        for (int b = 0; b < G::Blocks; ++b) mbar_init(&full[b], 1);
        for (int b = 0; b < kT * G::Depth; ++b) mbar_init(&done[b], R * G::Row);
        for (int b = 0; b < G::Outs; ++b) mbar_init(&freed[b], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // The launch before may still run from here on (a batch waits at once: that launch moves its clock).
    constexpr bool kEarly = !BATCH && G::Early;
    auto wait_for_grid = [] { asm volatile("griddepcontrol.wait;" ::: "memory"); };
    if (!kEarly) wait_for_grid();

    // A wait that gives up sets s_abort; every warp then leaves at its next wait.
    volatile int* abort_flag = &s_abort;
    auto wait = [&](uint64_t* bar, unsigned parity) -> bool {
        if (mbar_try_wait(bar, parity)) return true;
        const long long t0 = clock64();
        while (!mbar_try_wait(bar, parity)) {
            if (*abort_flag) return false;
            if (clock64() - t0 > kWaitCycles) {
                *abort_flag = 1;
                return false;
            }
        }
        return true;
    };
    // Iterations are numbered through all units of the CTA (`it0` before this one): iteration it of a
    // level completes phase it / Depth of done[level][it % Depth].
    struct Unit {
        int inst, i0, j0, j1, iters, a0;
    };
    auto args = [&](int inst) -> Args {
        if constexpr (BATCH)
            return p.desc[inst].a[p.parity];
        else
            return a_;
    };
    auto unit = [&](int u) {
        Unit t;
        if constexpr (BATCH) {
            const int4 v = p.units[u];
            t.inst = v.x;
            t.i0 = v.y;
            t.j0 = v.z;
            t.j1 = v.w;
        } else {
            const int strip = u % a_.strips, seg = u / a_.strips;
            t.inst = 0;
            t.i0 = strip * kX;
            t.j0 = seg * a_.seg_rows;
            t.j1 = min(t.j0 + a_.seg_rows, a_.lp.ny);
        }
        t.iters = (t.j1 - t.j0 + G::C + R - 1) / R;
        t.a0 = t.j0 + (kT - 1) * G::Lag - G::C;  // level 1's first row
        return t;
    };
    int u_first = blockIdx.x, u_end = 0, u_step = gridDim.x;
    long long step = 0;   // batch: the step of this launch, and its level n - 1 in the pulse tables
    int table_level = 0;
    if constexpr (BATCH) {
        u_first = p.first[blockIdx.x];
        u_end = p.first[blockIdx.x + 1];
        u_step = 1;
        step = const_cast<const volatile BatchClock*>(p.clk)->n;
        if (SRC == TRTR_SRC_PULSE) table_level = table_entry_at(p.clk, kT, p.flag);
    } else {
        u_end = a_.units;
    }

    if (w == G::Warps) {
        // The mover: lane 0 loads the blocks (block m of a unit: the rows a0 + 1 - R + m R ..; iteration
        // k needs the blocks up to k + 1) and stores the rows the last level has finished.
        unsigned phase = 0, it0 = 0, pending = 0;
        bool ok = true, fields_loaded = false;
        // block m of unit t: its populations, its fields
        auto load_populations = [&](const Unit& t, const SweepArgs& a, const CUtensorMap* mp, int m) {
            const unsigned b = (phase + m) % G::Blocks;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                int y = t.a0 + 1 - R + m * R + r;
                y = y < 0 ? y + a.lp.ny : (y >= a.lp.ny ? y - a.lp.ny : y);
                unsigned char* pd = smem + (b * R + r) * G::PopPitch;
                const int xp = t.i0 - 2 * kT + a.lp.gx;
                if (in_tile((int)(b * R) + r, G::Ring) && in_tile(y, a.lp.ny) && tma_ok(pd, xp, y, G::ES)) tma_load_3d(pd, mp, &full[b], xp, y + kGhostP, 0);
            }
        };
        auto load_fields = [&](const Unit& t, const SweepArgs& a, const CUtensorMap* mf, int m) {
            const unsigned b = (phase + m) % G::Blocks;
            mbar_expect_tx(&full[b], R * (G::PopRow + G::FldRow));
#pragma unroll
            for (int r = 0; r < R; ++r) {
                int y = t.a0 + 1 - R + m * R + r;
                y = y < 0 ? y + a.lp.ny : (y >= a.lp.ny ? y - a.lp.ny : y);
                unsigned char* fd = smem + G::FldOff + (b * R + r) * G::FldRow;
                const int xf = t.i0 - kT + a.gxf;
                if (tma_ok(fd, xf, y, 4)) tma_load_3d(fd, mf, &full[b], xf, y + a.gyf, 0);
            }
        };
        if constexpr (kEarly) {
            if (lane == 0) {
                prefetch_tensormap(&mp_);
                prefetch_tensormap(&mo_);
                if (u_first < u_end) {
                    const Unit t = unit(u_first);
                    for (int m = 0; m < min(t.iters + 1, 2 + G::Ahead); ++m) load_fields(t, a_, &mf_, m);
                }
            }
            fields_loaded = true;
            wait_for_grid();
        }
        for (int u = u_first; u < u_end && ok; u += u_step) {
            const Unit t = unit(u);
            Args a = args(t.inst);
            const CUtensorMap *mp, *mf, *mo;
            if constexpr (BATCH) {
                const SweepDesc* d = p.desc + t.inst;
                mp = &d->mp[p.parity];
                mf = &d->mf;
                mo = &d->mo[p.parity ^ 1];
            } else {
                mp = &mp_;
                mf = &mf_;
                mo = &mo_;
            }
            const int blocks = t.iters + 1;
            auto load = [&](int m) {
                load_fields(t, a, mf, m);
                load_populations(t, a, mp, m);
            };
            int loaded = min(blocks, 2 + G::Ahead);
            if (lane == 0)
                for (int m = 0; m < loaded; ++m) {
                    if (!fields_loaded) load_fields(t, a, mf, m);
                    load_populations(t, a, mp, m);
                }
            fields_loaded = false;
            for (int k = 0; k < t.iters; ++k) {
                const unsigned it = it0 + k, o = it % G::Outs;
                if (!(ok = wait(&done[(kT - 1) * G::Depth + it % G::Depth], (it / G::Depth) & 1))) break;
                const int y = t.a0 + k * R - (kT - 1) * G::Lag;  // the last level's rows
                unsigned char* buf = smem + G::OutOff + o * G::OutBytes;
                if (lane == 0) {
                    fence_proxy_async_smem();  // what the levels wrote in the ring and the buffer, for TMA
                    if (k + 2 + G::Ahead < blocks) load(k + 2 + G::Ahead);
                    if (y >= t.j0) tma_store_3d(mo, buf, t.i0, y, 0);
                    bulk_commit();
                }
                if (lane == 0) {  // the store before this one has left its buffer
                    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    if (it > 0) mbar_arrive(&freed[(it - 1) % G::Outs]);
                }
                loaded = min(blocks, k + 3 + G::Ahead);
            }
            pending = phase + loaded;
            phase += blocks;
            it0 += t.iters;
        }
        if (lane == 0) {
            // a wait gave up (the flag alone: the last level's for its last buffer): let the loads issued into
            // this CTA's shared memory land (bounded)
            if (!ok || *abort_flag) {
                if constexpr (BATCH)
                    atomicExch(p.flag, 1);
                else
                    atomicExch(a_.flag, 1);
                const unsigned n = pending < (unsigned)G::Blocks ? pending : (unsigned)G::Blocks;
                for (unsigned m = pending - n; m < pending; ++m)
                    mbar_wait_bounded(&full[m % G::Blocks], (m / G::Blocks) & 1);
            }
            bulk_wait_all();
            // every warp has read the clock: the last level has finished its units (or a wait gave up)
            if constexpr (BATCH) advance_clock(p.clk, kT);
        }
        return;
    }

    // Level `level`, row r0 of every iteration, its columns from 64 part on.
    const int level = w / (R * G::Row) + 1, r0 = w / G::Row % R, part = w % G::Row;
    uint32_t rkey = 0u;
    if constexpr (BATCH)
        rkey = RND != kRoundNearest ? sr_step_key((long)step + level - 1) : 0u;
    else
        rkey = a_.rkey[level - 1];
    unsigned phase = 0, it = 0;
    for (int u = u_first; u < u_end; u += u_step) {
        const Unit t = unit(u);
        Args a = args(t.inst);
        const int nx = a.lp.nx, ny = a.lp.ny;
        // per strip: the pairs' columns, their images for the rounding keys, their pulse factors
        const int i = t.i0 - kT + 2 * lane + 64 * part;
        F2 p1p[G::P], p2p[G::P], p1n[G::P], p2n[G::P];
        int wa[G::P], wb[G::P];
        uint32_t sel[G::P];
        const float* lev = a.pulse + (size_t)(table_level + level - 1) * a.pt.level;
#pragma unroll
        for (int h = 0; h < G::P; ++h) {
            if (SRC == TRTR_SRC_PULSE && in_tables(a.pt, i + 64 * h, 2, 0)) {
                p1p[h] = F2(__ldg(reinterpret_cast<const float2*>(lev + i + 64 * h)));
                p2p[h] = F2(__ldg(reinterpret_cast<const float2*>(lev + a.pt.p2 + i + 64 * h)));
                p1n[h] = F2(__ldg(reinterpret_cast<const float2*>(lev + a.pt.level + i + 64 * h)));
                p2n[h] = F2(__ldg(reinterpret_cast<const float2*>(lev + a.pt.level + a.pt.p2 + i + 64 * h)));
            }
            auto wrap = [&](int v) { return v < 0 ? v + nx : (v >= nx ? v - nx : v); };
            const int xa = wrap(i + 64 * h), xb = wrap(i + 64 * h + 1);
            wa[h] = xa & ~1;
            wb[h] = xb & ~1;
            sel[h] = (xa & 1 ? 0x32u : 0x10u) | (xb & 1 ? 0x7600u : 0x5400u);
        }
        const float* ty = lev + a.pt.y;

        if (kEarly && u == u_first) wait_for_grid();

        // the warp's row of the iteration and its ring row (block m = 0 starts at row a0 + 1 - R)
        int j = t.a0 - (level - 1) * G::Lag + r0;
        int ring = (int)(phase % G::Blocks) * R + j - (t.a0 + 1 - R);
        ring = ring < 0 ? ring + G::Ring : (ring >= G::Ring ? ring - G::Ring : ring);
        unsigned block = phase % G::Blocks, parity = (phase / G::Blocks) & 1;
        if (level == 1 && !wait(&full[block], parity)) return;
        // The row's pulse factors.  FP32 loads them an iteration ahead (4096^2: 102.5 -> 98.9 us a step; the 2-byte
        // storages, with more arithmetic in flight, lose 2 %).
        constexpr bool kAheadFactors = G::ES == 4;
        float2 qp = make_float2(0.f, 0.f), qn = qp;
        auto load_factors = [&](int y) {
            y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
            if (!in_tables(a.pt, 0, 1, y)) return;
            qp = __ldg(reinterpret_cast<const float2*>(ty + 2 * y));
            qn = __ldg(reinterpret_cast<const float2*>(ty + a.pt.level + 2 * y));
        };
        if (SRC == TRTR_SRC_PULSE && kAheadFactors) load_factors(j);
        for (int k = 0; k < t.iters; ++k, j += R, ++it) {
            F2 src[G::P];
#pragma unroll
            for (int h = 0; h < G::P; ++h) src[h] = F2(0.f);
            int yw = 0;
            if (RND != kRoundNearest) yw = j < 0 ? j + ny : (j >= ny ? j - ny : j);
            if (SRC == TRTR_SRC_PULSE) {  // as pulse_source_dt
                if (!kAheadFactors) load_factors(j);
#pragma unroll
                for (int h = 0; h < G::P; ++h)
                    src[h] = vfma(F2(1.5f), vfma(p1n[h], F2(qn.x), p2n[h] * F2(qn.y)),
                                  F2(-0.5f) * vfma(p1p[h], F2(qp.x), p2p[h] * F2(qp.y)));
                if (kAheadFactors) load_factors(j + R);
            }
            // level 1 waits for its rows, the others for the level before to have finished the iteration
            // before this one; the last level also, before it writes, for its output buffer
            bool ok;
            if (level == 1) {
                if (++block == G::Blocks) {
                    block = 0;
                    parity ^= 1;
                }
                ok = wait(&full[block], parity);
            } else {
                ok = it == 0 || wait(&done[(level - 2) * G::Depth + (it - 1) % G::Depth], ((it - 1) / G::Depth) & 1);
            }
            const unsigned o = it % G::Outs;
            if (!ok) return;
            if (j >= t.j0 - (kT - level) && j < t.j1 + (kT - level)) {
                const int below = ring >= level ? ring - level : ring - level + G::Ring;
                const int above = ring + level < G::Ring ? ring + level : ring + level - G::Ring;
                const int col = 2 * lane + 64 * part;  // its pairs, and the columns that they reach in the ring
                const bool inside = in_tile(below, G::Ring) && in_tile(ring, G::Ring) && in_tile(above, G::Ring) &&
                                    in_tile(col + kT - level, kW) && in_tile(col + kT + 64 * (G::P - 1) + 1 + level, kW) &&
                                    in_tile(col + 64 * (G::P - 1) + 1, kWC);
                constexpr int kPitch = G::PopPitch / G::ES;
                S* base = reinterpret_cast<S*>(smem) + 2 * lane + 64 * part + kT;
                S* pm = base + below * kPitch;
                S* p0 = base + ring * kPitch;
                S* pp = base + above * kPitch;
                const float* f = reinterpret_cast<const float*>(smem + G::FldOff) + ring * (G::NF * kWC) + 2 * lane + 64 * part;
                RoundKey rk[G::P] = {};
#pragma unroll
                for (int h = 0; h < G::P; ++h) {
                    if (RND != kRoundNearest) rk[h].a = sr_pair_key(wa[h], yw, nx, rkey);
                    if (RND == kRoundNodes) {
                        rk[h].b = sr_pair_key(wb[h], yw, nx, rkey);
                        rk[h].sel = sel[h];
                    }
                }
                S* buf = reinterpret_cast<S*>(smem + G::OutOff + o * G::OutBytes) + r0 * kX + 2 * lane + 64 * part - kT;
                auto buffer_free = [&]() { return it < (unsigned)G::Outs || wait(&freed[o], (it / G::Outs - 1) & 1); };
                if (inside) switch (level) {
                    case 1: sweep_row<S, 1, SRC, RND, G>(pm, p0, pp, f, src, a, rk, buf, lane, part, i, j, buffer_free); break;
                    case 2: sweep_row<S, 2, SRC, RND, G>(pm, p0, pp, f, src, a, rk, buf, lane, part, i, j, buffer_free); break;
                    case 3: sweep_row<S, 3, SRC, RND, G>(pm, p0, pp, f, src, a, rk, buf, lane, part, i, j, buffer_free); break;
                    default: sweep_row<S, 4, SRC, RND, G>(pm, p0, pp, f, src, a, rk, buf, lane, part, i, j, buffer_free); break;
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&done[(level - 1) * G::Depth + it % G::Depth]);
            ring += R;
            if (ring >= G::Ring) ring -= G::Ring;
        }
        phase += t.iters + 1;
    }
}

// The kGhostX ghost columns of every interior row and plane from the interior (periodic).
template <typename E>
__device__ __forceinline__ void refresh_ghost_columns(E* P, const PlaneLayout& L) {
    const int n = kQ * L.ny * 2 * kGhostX;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int g = k % (2 * kGhostX), row = k / (2 * kGhostX), q = row / L.ny, j = row - q * L.ny;
        E* p = P + (size_t)q * L.plane + (size_t)(j + kGhostP) * L.pitch + L.gx;
        const int to = g < kGhostX ? g - kGhostX : L.nx + g - kGhostX;
        const int from = g < kGhostX ? L.nx + to : to - L.nx;
        if (in_frame(L, to, j, kGhostX, 0) && in_frame(L, from, j, 0, 0)) p[to] = p[from];
    }
}
template <typename E>
__global__ void refresh_ghost_columns_kernel(E* P, PlaneLayout L) {
    refresh_ghost_columns(P, L);
}

// The arguments of one context: from buffer `from` into the other.
template <typename S>
SweepArgs sweep_args(const trtr_ctx* ctx, int from) {
    SweepArgs a;
    memset(static_cast<void*>(&a), 0, sizeof(a));
    a.pt = PulseTab::make(ctx->p.nx, ctx->p.ny);
    a.dst = ctx->pop[from ^ 1];
    a.lp = ctx->lp;
    a.gxf = ctx->lt.gx;
    a.gyf = ctx->lt.gy;
    a.strips = (ctx->p.nx + kX - 1) / kX;
    a.tau2_fixed = ctx->p.tau2_mode == TRTR_TAU2_FIXED;
    a.magic = (float)ctx->p.magic;
    a.omega2_fixed = (float)(ctx->p.tau2_mode == TRTR_TAU2_FIXED ? 1.0 / ctx->p.tau2 : 0.0);
    a.phi_ref = (float)ctx->p.phi_ref;
    return a;
}

template <typename S, int SRC, int RND>
cudaError_t launch_sweep_typed(trtr_ctx* ctx) {
    using G = Sweep<S, SRC>;
    auto kernel = sweep_kernel<S, SRC, RND, G, false>;
    static int configured_device = -1;
    if (configured_device != ctx->device) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, G::Smem);
        if (e != cudaSuccess) return e;
        configured_device = ctx->device;
    }
    SweepArgs a = sweep_args<S>(ctx, ctx->cur);
    a.pulse = SRC == TRTR_SRC_PULSE ? pulse_level<float>(ctx, a.pt, ctx->step) : nullptr;
    a.flag = ctx->dflag;
    a.seg_rows = ctx->sweep_rows;
    a.units = a.strips * ((ctx->p.ny + a.seg_rows - 1) / a.seg_rows);
    for (int s = 0; s < kT; ++s) a.rkey[s] = sr_step_key(ctx->step + s);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.units < ctx->num_sms ? a.units : ctx->num_sms));
    cfg.blockDim = dim3(G::Threads);
    cfg.dynamicSmemBytes = G::Smem;
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    if (G::Early) {  // not over the kernel that wrote what is read early
        attr[0].val.programmaticStreamSerializationAllowed = !ctx->tables_new;
        ctx->tables_new = false;
    }
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, ctx->maps4[ctx->cur], ctx->maps4[4], ctx->maps4[2 + (ctx->cur ^ 1)], a,
                              ManyGrids());
}

// The maps of one context: population rows (buffers 0, 1), interior stores (0, 1; whole 16-byte chunks of a
// row), field rows.
template <typename S, class G>
bool encode_maps_of(const trtr_ctx* ctx, CUtensorMap* rows, CUtensorMap* stores, CUtensorMap* fields) {
    bool ok = true;
    PlaneLayout in = ctx->lp;  // the interior alone, so that stores are clipped to it
    in.nx = bulk_cols_of<S>(in.nx);
    for (int b = 0; b < 2; ++b) {
        ok = ok && encode(&rows[b], tma_type<S>(), (int)sizeof(S), ctx->pop[b], ctx->lp, kQ, kW, 1, kQ);
        ok = ok && encode_interior(&stores[b], tma_type<S>(), (int)sizeof(S), ctx->pop[b], in, kQ, kX, G::R, kQ);
    }
    return ok && encode(fields, tma_type<float>(), 4, ctx->fld2, ctx->lt, G::NF, kWC, 1, G::NF);
}

// Rows of a segment: the number of segments a strip that ends soonest, by rounds of the SMs times a unit's
// rows (once per context: the search took longer than a launch of a 512^2 grid).  *iterations: of a CTA.
template <class G>
int segment_rows(const trtr_ctx* ctx, double* iterations) {
    const int ny = ctx->p.ny, strips = (ctx->p.nx + kX - 1) / kX;
    long best = 0;
    int best_rows = ny;
    for (int s = 1; s <= (ny + G::R - 1) / G::R && s <= 4 * ctx->num_sms; ++s) {
        const int rows = ((ny + s - 1) / s + G::R - 1) / G::R * G::R;
        const long units = (long)strips * ((ny + rows - 1) / rows);
        const long cost = ((units + ctx->num_sms - 1) / ctx->num_sms) * (rows + G::C + 4);
        if (s == 1 || cost < best) {
            best = cost;
            best_rows = rows;
        }
    }
    *iterations = (double)best / G::R;
    return best_rows;
}

template <typename S, int SRC>
cudaError_t encode4_typed(trtr_ctx* ctx) {
    // A strip costs its 128 columns however few of them the grid has, and a segment its ramp: grids of up to 32
    // columns (FP32) or of about 40 rows take longer than two two-step launches.  Measured (GB300, FP32 pulse, us for
    // four steps, sweep / two-step launches): 16 x 8000 33.7 / 26.8, 32 x 20000 73.2 / 69.2, 20000 x 32 42.8 / 34.5,
    // 48 x 8000 34.0 / 44.5, 121 x 1000 14.2 / 15.8, 4000 x 64 15.4 / 20.7, 500^2 14.9 / 22.7; without a source
    // 16 x 8000 26.6 / 24.8, 20000 x 32 34.0 / 31.8; FP16 20000 x 32 38.4 / 37.6, 16 x 8000 31.7 / 44.9.  Both sides are
    // estimated to 15 %, most within 8: the sweep has to win by that.
    double iterations = 0.0;
    ctx->sweep_rows = segment_rows<Sweep<S, SRC>>(ctx, &iterations);
    ctx->sweep_sooner = 1.08 * sweep_us(ctx->p.precision, ctx->p.src_mode, iterations) <
                        2.0 * two_step_us(ctx->p.precision, ctx->p.src_mode, ctx->num_sms, ctx->p.nx, ctx->p.ny);
    return encode_maps_of<S, Sweep<S, SRC>>(ctx, &ctx->maps4[0], &ctx->maps4[2], &ctx->maps4[4]) ? cudaSuccess
                                                                                                 : cudaErrorInvalidValue;
}

// ---- batches -------------------------------------------------------------------------------------

// The four ghost columns of every instance's current buffer.
template <typename E>
__global__ void batch_ghost_columns_kernel(const SweepDesc* desc, int parity) {
    const SweepDesc& d = desc[blockIdx.y];
    refresh_ghost_columns(static_cast<E*>(d.pop[parity]), d.a[0].lp);
}

// The work-list: strips cut into segments of at most most_rows rows, the units dealt longest first to the CTA with
// the least work so far.  Returns the rows (ramps included) of the busiest CTA; with lists, also the units
// in the CTAs' order.
struct Unit {
    int rows, cta;
    int4 at;
};
template <class G>
long deal_units(trtr_ctx* const* ctx, int count, int ctas, long most_rows, std::vector<Unit>& all, std::vector<int4>* units,
                std::vector<int>* first) {
    all.clear();
    for (int k = 0; k < count; ++k) {
        const int nx = ctx[k]->p.nx, ny = ctx[k]->p.ny;
        const int segs = (int)((ny + most_rows - 1) / most_rows);
        const int rows = ((ny + segs - 1) / segs + G::R - 1) / G::R * G::R;
        for (int j0 = 0; j0 < ny; j0 += rows)
            for (int i0 = 0; i0 < nx; i0 += kX) {
                const int j1 = std::min(j0 + rows, ny);
                all.push_back(Unit{j1 - j0 + G::C + 4, 0, make_int4(k, i0, j0, j1)});
            }
    }
    std::stable_sort(all.begin(), all.end(), [](const Unit& a, const Unit& b) { return a.rows > b.rows; });
    using Load = std::pair<long, int>;
    std::vector<Load> heap(ctas);
    for (int c = 0; c < ctas; ++c) heap[c] = {0, c};
    std::priority_queue<Load, std::vector<Load>, std::greater<Load>> load(std::greater<Load>(), std::move(heap));
    long busiest = 0;
    for (Unit& u : all) {
        Load l = load.top();
        load.pop();
        u.cta = l.second;
        l.first += u.rows;
        busiest = std::max(busiest, l.first);
        load.push(l);
    }
    if (units) {
        first->assign(ctas + 1, 0);
        for (const Unit& u : all) ++(*first)[u.cta + 1];
        for (int c = 0; c < ctas; ++c) (*first)[c + 1] += (*first)[c];
        std::vector<int> next(first->begin(), first->end() - 1);
        units->resize(all.size());
        for (const Unit& u : all) (*units)[next[u.cta]++] = u.at;
    }
    return busiest;
}

template <typename S>
cudaError_t setup_batch_typed(trtr_ctx* const* ctx, int count, cudaStream_t stream, SweepBatch* out) {
    using G = Sweep<S, TRTR_SRC_NONE>;  // (the pulse's is the same)
    static_assert(Sweep<S, TRTR_SRC_PULSE>::R == G::R && Sweep<S, TRTR_SRC_PULSE>::NF == G::NF, "one geometry");
    const int ctas = ctx[0]->num_sms;
    long total = 0;
    for (int k = 0; k < count; ++k) total += (long)((ctx[k]->p.nx + kX - 1) / kX) * ctx[k]->p.ny;
    std::vector<Unit> scratch;
    std::vector<int4> best_units;
    std::vector<int> best_first;
    long best = -1, best_rows = 0, last_rows = 0;
    for (int parts = 1; parts <= 6; ++parts) {
        const long rows = std::max((long)G::R * 2, total / ((long)ctas * parts) + 1);
        if (rows == last_rows) continue;
        last_rows = rows;
        const long busiest = deal_units<G>(ctx, count, ctas, rows, scratch, nullptr, nullptr);
        if (best < 0 || busiest < best) {
            best = busiest;
            best_rows = rows;
        }
    }
    deal_units<G>(ctx, count, ctas, best_rows, scratch, &best_units, &best_first);
    out->rows = best;
    out->iteration_rows = G::R;
    std::vector<SweepDesc> h(count);
    for (int k = 0; k < count; ++k) {
        const trtr_ctx* c = ctx[k];
        SweepDesc& d = h[k];
        if (!encode_maps_of<S, G>(c, d.mp, d.mo, &d.mf)) return cudaErrorInvalidValue;
        for (int b = 0; b < 2; ++b) {
            d.a[b] = sweep_args<S>(c, b);
            d.a[b].pulse = c->ptab ? static_cast<const float*>(c->ptab) + kTabGhost : nullptr;
            d.pop[b] = c->pop[b];
        }
    }
    out->ctas = ctas;
    const size_t desc_bytes = sizeof(SweepDesc) * count, unit_bytes = sizeof(int4) * best_units.size();
    const size_t first_bytes = sizeof(int) * best_first.size();
    std::vector<char> all(desc_bytes + unit_bytes + first_bytes);
    memcpy(all.data(), h.data(), desc_bytes);
    memcpy(all.data() + desc_bytes, best_units.data(), unit_bytes);
    memcpy(all.data() + desc_bytes + unit_bytes, best_first.data(), first_bytes);
    cudaError_t e = cudaMalloc(&out->d_desc, all.size());
    if (e != cudaSuccess) return e;
    out->d_units = static_cast<char*>(out->d_desc) + desc_bytes;
    out->d_first = static_cast<char*>(out->d_units) + unit_bytes;
    e = cudaMemcpyAsync(out->d_desc, all.data(), all.size(), cudaMemcpyHostToDevice, stream);
    const cudaError_t s = cudaStreamSynchronize(stream);  // the vector goes out of scope
    return e != cudaSuccess ? e : s;
}

template <typename S, int SRC, int RND>
cudaError_t launch_batch_typed(const SweepBatch& b, BatchClock* clk, int* flag, int parity, cudaStream_t stream) {
    using G = Sweep<S, SRC>;
    auto kernel = sweep_kernel<S, SRC, RND, G, true>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, G::Smem);
    if (e != cudaSuccess) return e;
    ManyGrids p;
    p.desc = static_cast<const SweepDesc*>(b.d_desc);
    p.units = static_cast<const int4*>(b.d_units);
    p.first = static_cast<const int*>(b.d_first);
    p.clk = clk;
    p.flag = flag;
    p.parity = parity;
    kernel<<<b.ctas, G::Threads, G::Smem, stream>>>(CUtensorMap(), CUtensorMap(), CUtensorMap(), SweepArgs(), p);
    return cudaGetLastError();
}

}  // namespace

// Rows wrap once around the grid, and a row holds at least one whole 16-byte chunk.
static bool sweep_size(const trtr_ctx* ctx) { return ctx->p.nx >= 16 && ctx->p.ny >= 32; }

// Fitted to launches of 5 to 140 iterations on GB300 (FP32 to 6 %, FP16 to 13 %; the first iterations, which only
// load, are shorter): us an iteration of three rows (two with a source field; four of the 2-byte storages).
double sweep_us(int precision, int src, double iterations) {
    if (precision != TRTR_F32) return src == TRTR_SRC_PULSE ? 2.1 * iterations - 5.0 : 1.8 * iterations - 3.6;
    const double us = src == TRTR_SRC_PULSE ? 1.40 : (src == TRTR_SRC_FIELD ? 0.89 : 1.13);
    return us * iterations - 1.8;
}

cudaError_t encode_maps4(trtr_ctx* ctx) {
    if (!ctx->fld2 || !sweep_size(ctx)) return cudaSuccess;
    const bool field = ctx->p.src_mode == TRTR_SRC_FIELD;
    switch (ctx->p.precision) {
        case TRTR_F32: return field ? encode4_typed<float, TRTR_SRC_FIELD>(ctx) : encode4_typed<float, TRTR_SRC_NONE>(ctx);
        case TRTR_F16_OFS:
            return field ? encode4_typed<__half, TRTR_SRC_FIELD>(ctx) : encode4_typed<__half, TRTR_SRC_NONE>(ctx);
        case TRTR_BF16_OFS:
            return field ? encode4_typed<__nv_bfloat16, TRTR_SRC_FIELD>(ctx) : encode4_typed<__nv_bfloat16, TRTR_SRC_NONE>(ctx);
        default: return cudaErrorInvalidValue;
    }
}

// Source fields: while S^n is S^{n-1}, so that every step of the launch has the same source term.
bool sweep_applies(const trtr_ctx* ctx) {
    if (!ctx->fld2 || ctx->steps_per_launch != 2 || ctx->p.bc_mode != TRTR_BC_PERIODIC || !sweep_size(ctx)) return false;
    return ctx->p.src_mode != TRTR_SRC_FIELD || ctx->S_prev < 0 || ctx->S_prev == ctx->S_cur;
}

// The source term of a stationary field, with the one-step kernel's roundings of 1.5 S - 0.5 S, at every
// node of the packed fields' ghost frame.
__global__ void pack_source_kernel(float* dst, const float* S, PlaneLayout lt, PlaneLayout lf) {
    const unsigned gw = lt.nx + 2 * kGhostT, n = gw * (unsigned)(lt.ny + 2 * kGhostT);
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int j = (int)(k / gw) - kGhostT, i = (int)(k % gw) - kGhostT;
        const float s = S[lf.at((i % lt.nx + lt.nx) % lt.nx, (j % lt.ny + lt.ny) % lt.ny)];
        dst[lt.at(i, j)] = __fmaf_rn(1.5f, s, __fmul_rn(-0.5f, s));
    }
}

cudaError_t launch_pack_source(trtr_ctx* ctx) {
    const unsigned n = (unsigned)(ctx->p.nx + 2 * kGhostT) * (unsigned)(ctx->p.ny + 2 * kGhostT);
    const unsigned want = (n + 255) / 256, cap = (unsigned)ctx->num_sms * 8;
    ctx->launches += 1;
    ctx->tables_new = true;
    pack_source_kernel<<<want < cap ? want : cap, 256, 0, ctx->stream>>>(
        static_cast<float*>(ctx->fld2) + 5 * ctx->lt.plane,
        static_cast<const float*>(ctx->S) + (size_t)ctx->S_cur * ctx->lf.plane, ctx->lt, ctx->lf);
    return cudaGetLastError();
}

cudaError_t launch_ghost_columns(trtr_ctx* ctx) {
    const int n = kQ * ctx->p.ny * 2 * kGhostX, want = (n + 255) / 256, cap = ctx->num_sms * 4;
    ctx->launches += 1;
    if (ctx->esize == 4)
        refresh_ghost_columns_kernel<<<want < cap ? want : cap, 256, 0, ctx->stream>>>(
            static_cast<float*>(ctx->pop[ctx->cur]), ctx->lp);
    else
        refresh_ghost_columns_kernel<<<want < cap ? want : cap, 256, 0, ctx->stream>>>(
            static_cast<unsigned short*>(ctx->pop[ctx->cur]), ctx->lp);
    return cudaGetLastError();
}

template <typename S, int RND>
static cudaError_t launch_sweep_src(trtr_ctx* ctx) {
    switch (ctx->p.src_mode) {
        case TRTR_SRC_FIELD: return launch_sweep_typed<S, TRTR_SRC_FIELD, RND>(ctx);
        case TRTR_SRC_PULSE: return launch_sweep_typed<S, TRTR_SRC_PULSE, RND>(ctx);
        default: return launch_sweep_typed<S, TRTR_SRC_NONE, RND>(ctx);
    }
}

template <typename S>
static cudaError_t launch_sweep_2byte(trtr_ctx* ctx) {
    if (ctx->p.rounding != TRTR_ROUND_STOCHASTIC) return launch_sweep_src<S, kRoundNearest>(ctx);
    return ctx->p.nx % 2 == 0 ? launch_sweep_src<S, kRoundPairs>(ctx) : launch_sweep_src<S, kRoundNodes>(ctx);
}

cudaError_t launch_sweep(trtr_ctx* ctx) {
    switch (ctx->p.precision) {
        case TRTR_F32: return launch_sweep_src<float, kRoundNearest>(ctx);
        case TRTR_F16_OFS: return launch_sweep_2byte<__half>(ctx);
        case TRTR_BF16_OFS: return launch_sweep_2byte<__nv_bfloat16>(ctx);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t sweep_batch_setup(trtr_ctx* const* ctx, int count, cudaStream_t stream, SweepBatch* out) {
    switch (ctx[0]->p.precision) {
        case TRTR_F32: return setup_batch_typed<float>(ctx, count, stream, out);
        case TRTR_F16_OFS: return setup_batch_typed<__half>(ctx, count, stream, out);
        case TRTR_BF16_OFS: return setup_batch_typed<__nv_bfloat16>(ctx, count, stream, out);
        default: return cudaErrorInvalidValue;
    }
}

void sweep_batch_free(SweepBatch* b) {
    if (b->d_desc) cudaFree(b->d_desc);
    *b = SweepBatch();
}

cudaError_t sweep_batch_ghost_columns(const SweepBatch& b, int count, int esize, int parity, cudaStream_t stream) {
    for (int k = 0; k < count; k += 65535) {
        const SweepDesc* d = static_cast<const SweepDesc*>(b.d_desc) + k;
        const dim3 grid(16, count - k < 65535 ? count - k : 65535);
        if (esize == 4)
            batch_ghost_columns_kernel<float><<<grid, 256, 0, stream>>>(d, parity);
        else
            batch_ghost_columns_kernel<unsigned short><<<grid, 256, 0, stream>>>(d, parity);
    }
    return cudaGetLastError();
}

template <typename S, int RND>
static cudaError_t launch_batch_src(const SweepBatch& b, BatchClock* clk, int* flag, int parity, int src, cudaStream_t stream) {
    return src == TRTR_SRC_PULSE ? launch_batch_typed<S, TRTR_SRC_PULSE, RND>(b, clk, flag, parity, stream)
                                 : launch_batch_typed<S, TRTR_SRC_NONE, RND>(b, clk, flag, parity, stream);
}
template <typename S>
static cudaError_t launch_batch_2byte(const SweepBatch& b, BatchClock* clk, int* flag, int parity, int src, bool sr, bool odd,
                                      cudaStream_t stream) {
    if (!sr) return launch_batch_src<S, kRoundNearest>(b, clk, flag, parity, src, stream);
    return odd ? launch_batch_src<S, kRoundNodes>(b, clk, flag, parity, src, stream)
               : launch_batch_src<S, kRoundPairs>(b, clk, flag, parity, src, stream);
}

cudaError_t sweep_batch_launch(const SweepBatch& b, BatchClock* clk, int* flag, int parity, int precision, int src, bool sr,
                               bool odd, cudaStream_t stream) {
    switch (precision) {
        case TRTR_F32: return launch_batch_src<float, kRoundNearest>(b, clk, flag, parity, src, stream);
        case TRTR_F16_OFS: return launch_batch_2byte<__half>(b, clk, flag, parity, src, sr, odd, stream);
        case TRTR_BF16_OFS: return launch_batch_2byte<__nv_bfloat16>(b, clk, flag, parity, src, sr, odd, stream);
        default: return cudaErrorInvalidValue;
    }
}

TRTR_BOUNDS_TAKE(sweep)

}  // namespace trtr
