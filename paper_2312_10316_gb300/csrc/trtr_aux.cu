// trtr_aux.cu -- kernels around the step: coefficient fields (with their ghost cells),
// the pulse closed form, equilibrium initialisation (shifted into the pull layout), the
// phi moment, the FP64 reductions (mass, RMS / relative L2 error of Eq. (33)) and
// population I/O.
#include <math.h>

#include <type_traits>

#include "trtr_step_core.cuh"

namespace trtr {

PlaneLayout make_layout(int nx, int ny, int elem_bytes, int ghost) {
    PlaneLayout L;
    L.nx = nx;
    L.ny = ny;
    const int line = 128 / elem_bytes;  // elements per 128-byte line
    L.gx = line;
    L.gy = ghost;
    long long pitch = ((long long)nx + 2LL * line + line - 1) / line * line;
    if (pitch < 320) pitch = 320;  // wider than every TMA box (<= 256 elements + origin shift)
    L.pitch = (int)pitch;
    L.rows = ny + 2 * ghost < 16 ? 16 : ny + 2 * ghost;
    L.plane = (size_t)L.rows * (size_t)L.pitch;
    return L;
}

namespace {

using core::weight;
constexpr int kThreads = 256;

// The kernels of a time loop are launched with programmatic dependent launch: set up while the kernel
// before them still runs, they wait here for its completion before they touch memory.
__device__ __forceinline__ void overlap_launch() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ int wrap(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// Value of a field at ghosted position (i, j), i in [-1, nx], j in [-1, ny], from its interior
// values f(i, j): periodic wrap, or the linear extrapolation 2 f(edge) - f(edge -+ 1) (grad
// mode one-sided; a single node repeats itself).  Corners compose the two rules.
template <typename F>
__device__ __forceinline__ double ghosted(const F& f, int i, int j, int nx, int ny, int grad_mode) {
    auto along_x = [&](int jj) -> double {
        if (i >= 0 && i < nx) return f(i, jj);
        if (grad_mode == TRTR_GRAD_PERIODIC || nx == 1) return f(wrap(i, nx), jj);
        return i < 0 ? 2.0 * f(0, jj) - f(1, jj) : 2.0 * f(nx - 1, jj) - f(nx - 2, jj);
    };
    if (j >= 0 && j < ny) return along_x(j);
    if (grad_mode == TRTR_GRAD_PERIODIC || ny == 1) return along_x(wrap(j, ny));
    return j < 0 ? 2.0 * along_x(0) - along_x(1) : 2.0 * along_x(ny - 1) - along_x(ny - 2);
}

// u (with ghosts) and D from caller arrays [ny][nx] in physical units.
template <typename C>
__global__ void convert_fields_kernel(C* uv, C* Dh, const double* sux, const double* suy, const double* sD,
                                      PlaneLayout L, int grad_mode, double u_scale, double d_scale, double dh_const,
                                      int use_const) {
    const int gw = L.nx + 2, gh = L.ny + 2;
    const size_t n = (size_t)gw * gh;
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
        const int j = (int)(k / gw) - 1, i = (int)(k % gw) - 1;
        auto fx = [&](int ii, int jj) { return sux[(size_t)jj * L.nx + ii]; };
        auto fy = [&](int ii, int jj) { return suy[(size_t)jj * L.nx + ii]; };
        uv[L.at(i, j)] = C(ghosted(fx, i, j, L.nx, L.ny, grad_mode) * u_scale);
        uv[L.plane + L.at(i, j)] = C(ghosted(fy, i, j, L.nx, L.ny, grad_mode) * u_scale);
        if (i >= 0 && i < L.nx && j >= 0 && j < L.ny)
            Dh[L.at(i, j)] = C(use_const ? dh_const : sD[(size_t)j * L.nx + i] * d_scale);
    }
}

template <typename C>
__global__ void pulse_fields_kernel(C* uv, C* Dh, C* tab_x, C* tab_y, PlaneLayout L, int grad_mode, double x0,
                                    double y0, double dx, double dt, Pulse pp, double dh_const, int use_const) {
    const int gw = L.nx + 2, gh = L.ny + 2;
    const size_t n = (size_t)gw * gh;
    const double us = dt / dx, ds = dt / (dx * dx);
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
        const int j = (int)(k / gw) - 1, i = (int)(k % gw) - 1;
        auto fx = [&](int ii, int jj) { return -pp.omega * (y0 + jj * dx); };
        auto fy = [&](int ii, int jj) { return pp.omega * (x0 + ii * dx); };
        uv[L.at(i, j)] = C(ghosted(fx, i, j, L.nx, L.ny, grad_mode) * us);
        uv[L.plane + L.at(i, j)] = C(ghosted(fy, i, j, L.nx, L.ny, grad_mode) * us);
        if (i < 0 || i >= L.nx || j < 0 || j >= L.ny) continue;
        const double x = x0 + i * dx, y = y0 + j * dx;
        Dh[L.at(i, j)] = C(use_const ? dh_const : pp.D0 * (1.0 + pp.D_amp * sin(M_PI * x) * sin(M_PI * y)) * ds);
        auto axis = [](C* tab, int n, int at, double v) {
            tab[at] = C(sin(M_PI * v));
            tab[n + at] = C(cos(M_PI * v));
            tab[2 * n + at] = C(v);
            tab[3 * n + at] = C(v - (double)C(v));
        };
        if (j == 0) axis(tab_x, L.nx, i, x);
        if (i == 0) axis(tab_y, L.ny, j, y);
    }
}

template <typename C>
__global__ void convert_source_kernel(C* dst, const double* S, PlaneLayout L, double dt) {
    overlap_launch();
    const unsigned n = (unsigned)L.nx * L.ny;
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int j = (int)(k / L.nx), i = (int)(k - (unsigned)j * L.nx);
        dst[L.at(i, j)] = C(dt * S[k]);
    }
}

__device__ __forceinline__ double pulse_phi(const PulseTime& pt, double x, double y) {
    const double rx = x - pt.cx, ry = y - pt.cy;
    return pt.amp * exp(-0.5 * (rx * rx + ry * ry) * pt.inv_s2);
}

// Third-order Hermite equilibrium (Eq. (6)) in lattice units, in FP64:
// w_i phi [1 + 3 eu + 4.5 ((eu)^2 - |u|^2/3) + 4.5 ((eu)^3 - eu |u|^2)], eu = e_i . uhat.
template <typename T>
__device__ __forceinline__ T equilibrium(int q, T phi, T u, T v) {
    const T eu = T(lattice_ex(q)) * u + T(lattice_ey(q)) * v;
    const T uu = u * u + v * v;
    return weight<T>(q) * phi *
           (T(1) + T(3) * eu + T(4.5) * (eu * eu - uu / T(3)) + T(4.5) * (eu * eu * eu - eu * uu));
}

// Stores value v of population q that node (i, j) pulls, P_q(x - e_q), periodic images included.
template <typename S>
__device__ __forceinline__ void store_pulled(S* P, const PlaneLayout& L, int q, int i, int j, bool inner, S v) {
    S* plane = P + q * L.plane;
    if (inner)  // the slot and its neighbours are away from the ghost frame
        plane[L.at(i - lattice_ex(q), j - lattice_ey(q))] = v;
    else
        store_with_ghosts(plane, L, wrap(i - lattice_ex(q), L.nx), wrap(j - lattice_ey(q), L.ny), v);
}
__device__ __forceinline__ bool inner_node(const PlaneLayout& L, int i, int j) {
    return i > L.gy && i < L.nx - 1 - L.gy && j > L.gy && j < L.ny - 1 - L.gy;
}

// Initial condition g_i(x) = g_i^eq(phi0(x), u(x)) in the pull layout: node x takes its nine equilibria in
// the compute type and stores g_i(x) where x pulls it, P_i(x - e_i), periodic images included (each slot
// has exactly one writer).
template <typename S, typename C>
__device__ __forceinline__ void init_node(S* P, const C* uv, const PlaneLayout& lp, const PlaneLayout& lf, int i, int j, C phi,
                                          C phi_ref) {
    const C u = uv[lf.at(i, j)], v = uv[lf.plane + lf.at(i, j)];
    const bool inner = inner_node(lp, i, j);
#pragma unroll
    for (int q = 0; q < kQ; ++q)
        store_pulled(P, lp, q, i, j, inner, Store<S>::encode(equilibrium<C>(q, phi, u, v), weight<C>(q) * phi_ref));
}

// From the caller's phi0: a node a thread (GB300, us, with 26 rows of a column a thread / now: FP32 2048^2
// 104 / 77, 40 x 4000 16.6 / 10.4).
template <typename S, typename C>
__global__ void __launch_bounds__(kThreads)
    init_eq_kernel(S* P, const C* uv, const double* phi0, PlaneLayout lp, PlaneLayout lf, C phi_ref) {
    const unsigned n = (unsigned)lp.nx * lp.ny;
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int j = (int)(k / lp.nx), i = (int)(k - (unsigned)j * lp.nx);
        init_node<S, C>(P, uv, lp, lf, i, j, (C)phi0[k], phi_ref);
    }
}

// The pulse at t = 0, the product of a factor of x and one of y, each taken once a block (w columns, `rows` rows):
// an FP64 exponential a node is 45 FP64 instructions and made this kernel 0.9 ms at 4096^2.
constexpr int kInitRows = 32, kInitThreads = 128;
template <typename S, typename C>
__global__ void __launch_bounds__(kInitThreads)
    init_pulse_kernel(S* P, const C* uv, PlaneLayout lp, PlaneLayout lf, double x0, double y0, double dx, PulseTime pt,
                      C phi_ref, int log_w, int rows) {
    __shared__ double f[kInitThreads + kInitRows];
    const int w = 1 << log_w, tid = threadIdx.x, i0 = blockIdx.x << log_w, j0 = blockIdx.y * rows;
    for (int t = tid; t < w + rows; t += kInitThreads) {
        const double r = t < w ? x0 + (i0 + t) * dx - pt.cx : y0 + (j0 + t - w) * dx - pt.cy;
        f[t] = (t < w ? pt.amp : 1.0) * exp(-0.5 * r * r * pt.inv_s2);
    }
    __syncthreads();
    const int c = tid & (w - 1), i = i0 + c;
    if (i >= lp.nx) return;
    for (int r = tid >> log_w; r < rows && j0 + r < lp.ny; r += kInitThreads >> log_w)
        init_node<S, C>(P, uv, lp, lf, i, j0 + r, (C)(f[c] * f[w + r]), phi_ref);
}

// Dirichlet boundary by non-equilibrium extrapolation (Sec. 3) over the buffer P that a step
// has just written.  For edge node b and its inward neighbour f (diagonal at corners):
//   g_i(b) = g_i^eq(phi_b, u_b) + g_i(f) - g_i^eq(phi(f), u_f),  g_i(f) = P_i(f - e_i),
// stored where b pulls it, P_i(b - e_i) (a ghost cell when b - e_i is outside the grid).  A
// slot P_i(y) is pulled by the node y + e_i alone, so the slots written here (pulled by edge
// nodes) and the slots read (pulled by interior nodes f) are disjoint: no thread ordering.
// One thread per edge node and population (threads of a warp share the population), in blocks of one
// warp: a node's 18 equilibria are 250 FP64 instructions, which on the two SMs of two 256-thread blocks
// took 20.7 us for the 400 edge nodes of a 101^2 grid, and one population's are 35.
template <typename S, typename C>
__global__ void dirichlet_nee_kernel(S* P, const C* uv, const double* phib, PlaneLayout lp, PlaneLayout lf,
                                     C phi_ref) {
    overlap_launch();
    const int nx = lp.nx, ny = lp.ny, nb = edge_count(nx, ny);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < kQ * nb; e += gridDim.x * blockDim.x) {
        const int q = e / nb, k = e - q * nb;
        int i, j;
        edge_node(k, nx, ny, &i, &j);
        const int fi = i == 0 ? 1 : (i == nx - 1 ? nx - 2 : i);
        const int fj = j == 0 ? 1 : (j == ny - 1 ? ny - 2 : j);
        double gq = 0.0, phif = 0.0;
#pragma unroll
        for (int p = 0; p < kQ; ++p) {
            const double gf = (double)Store<S>::decode(P[p * lp.plane + lp.at(fi - lattice_ex(p), fj - lattice_ey(p))],
                                                       weight<C>(p) * phi_ref);
            phif += gf;
            if (p == q) gq = gf;
        }
        const double ub = (double)uv[lf.at(i, j)], vb = (double)uv[lf.plane + lf.at(i, j)];
        const double uf = (double)uv[lf.at(fi, fj)], vf = (double)uv[lf.plane + lf.at(fi, fj)];
        const double g = equilibrium(q, phib[k], ub, vb) + gq - equilibrium(q, phif, uf, vf);
        P[q * lp.plane + lp.at(i - lattice_ex(q), j - lattice_ey(q))] = Store<S>::encode((C)g, weight<C>(q) * phi_ref);
    }
}

__global__ void gather_edges_kernel(double* phib, const double* phi, int nx, int ny) {
    overlap_launch();
    const int nb = edge_count(nx, ny);
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nb; k += gridDim.x * blockDim.x) {
        int i, j;
        edge_node(k, nx, ny, &i, &j);
        phib[k] = phi[(size_t)j * nx + i];
    }
}

// g_i(x, t_n) = P_i(x - e_i), decoded to the compute type.  x - e_i may be a ghost cell: it
// holds the periodic image, or the Dirichlet pass's value (TRTR_BC_DIRICHLET_NEE).
template <typename S, typename C>
__device__ __forceinline__ C pulled(const S* P, int q, int i, int j, const PlaneLayout& L, C phi_ref) {
    return Store<S>::decode(P[q * L.plane + L.at(i - lattice_ex(q), j - lattice_ey(q))], weight<C>(q) * phi_ref);
}

template <typename S, typename C>
__device__ __forceinline__ double node_phi(const S* P, int i, int j, const PlaneLayout& L, C phi_ref) {
    double phi = 0.0;
#pragma unroll
    for (int q = 0; q < kQ; ++q) phi += (double)pulled<S, C>(P, q, i, j, L, phi_ref);
    return phi;
}

// The FP32-computing storages: phi of the node pair (i, i + 1) as an unevaluated sum s + c + t of floats,
// exact to beyond FP64 (two levels of Knuth's error-free two-sum).  Converting the nine floats to
// FP64 and adding them there takes 17 instructions of the FP64 pipe (16 cycles each), which held
// these kernels at 36 G nodes/s; s + c + t leaves 5 of them.
using core::F2;
struct PhiPair {
    F2 s, c, t;
};
__device__ __forceinline__ F2 two_sum(F2 a, F2 b, F2& e) {
    const F2 s = a + b, bb = s - a;
    e = (a - (s - bb)) + (b - bb);
    return s;
}
template <typename S>
__device__ __forceinline__ void pulled_pair(const S* P, int i, int j, const PlaneLayout& L, float phi_ref, F2 g[kQ]) {
    using S2 = typename core::Pair<S>::type;
    const S* at = P + L.at(i, j);
    const bool ok = in_frame(L, i - 1, j - 1, kGhostP, kGhostP) && in_frame(L, i + 2, j + 1, kGhostP, kGhostP);
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        if (!ok) {
            g[q] = F2(0.f);
            continue;
        }
        const S* p = at + q * L.plane - (ptrdiff_t)lattice_ey(q) * L.pitch - lattice_ex(q);
        const float off = core::weight<float>(q) * phi_ref;
        g[q] = lattice_ex(q) == 0 ? core::Pair<S>::decode(*reinterpret_cast<const S2*>(p), off)
                                  : core::Pair<S>::decode(p[0], p[1], off);
    }
}
template <typename S>
__device__ __forceinline__ PhiPair pair_phi(const S* P, int i, int j, const PlaneLayout& L, float phi_ref) {
    F2 g[kQ];
    pulled_pair(P, i, j, L, phi_ref, g);
    PhiPair r;
    r.s = two_sum(g[0], g[1], r.c);
    r.t = F2(0.f);
#pragma unroll
    for (int q = 2; q < kQ; ++q) {
        F2 e, ee;
        r.s = two_sum(r.s, g[q], e);
        r.c = two_sum(r.c, e, ee);
        r.t = r.t + ee;
    }
    return r;
}
// The value in FP64; sums near the end of the float range (and beyond it, infinities and NaN) are
// taken in FP64 from the populations.
__device__ __forceinline__ bool float_sum_ok(float s) { return fabsf(s) < 1e36f; }
template <typename S>
__device__ __forceinline__ double phi_value(float s, float c, float t, const S* P, int i, int j, const PlaneLayout& L,
                                            float phi_ref) {
    return float_sum_ok(s) ? (double)s + ((double)c + (double)t) : node_phi<S, float>(P, i, j, L, phi_ref);
}

// The kernels that a host call waits for put the step kernels' timeout flag into its pinned copy.
__device__ __forceinline__ void report_flag(const int* flag, int* host_flag) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *host_flag = *flag;
}

template <typename S, typename C>
__global__ void __launch_bounds__(kThreads)
    moments_kernel(double* out, const S* P, PlaneLayout L, C phi_ref, const int* flag, int* host_flag) {
    overlap_launch();
    report_flag(flag, host_flag);
    if constexpr (sizeof(S) == 8) {
        const unsigned n = (unsigned)L.nx * L.ny;
        for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
            const int j = (int)(k / L.nx), i = (int)(k - (unsigned)j * L.nx);
            out[k] = node_phi<S, C>(P, i, j, L, phi_ref);
        }
    } else {
        const unsigned np = (L.nx + 1) / 2, n = np * L.ny;
        const bool wide = L.nx % 2 == 0 && (reinterpret_cast<uintptr_t>(out) & 15u) == 0u;
        for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
            const int j = (int)(k / np), i = 2 * (int)(k - (unsigned)j * np);
            const PhiPair p = pair_phi(P, i, j, L, phi_ref);
            double* o = out + (size_t)j * L.nx + i;
            const double a = phi_value(p.s.v.x, p.c.v.x, p.t.v.x, P, i, j, L, phi_ref);
            if (i + 1 < L.nx) {
                const double b = phi_value(p.s.v.y, p.c.v.y, p.t.v.y, P, i + 1, j, L, phi_ref);
                if (wide) {
                    *reinterpret_cast<double2*>(o) = make_double2(a, b);
                } else {
                    o[0] = a;
                    o[1] = b;
                }
            } else {
                o[0] = a;
            }
        }
    }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Deterministic two-value block sum (fixed tree); result valid in thread 0.
__device__ __forceinline__ void block_sum2(double& a, double& b) {
    __shared__ double sa[kThreads / 32], sb[kThreads / 32];
    a = warp_sum(a);
    b = warp_sum(b);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) {
        sa[w] = a;
        sb[w] = b;
    }
    __syncthreads();
    if (w == 0) {
        a = lane < kThreads / 32 ? sa[lane] : 0.0;
        b = lane < kThreads / 32 ? sb[lane] : 0.0;
        a = warp_sum(a);
        b = warp_sum(b);
    }
}

// A thread's part of a reduction of kind KIND:
//  kReduceMass: sum phi;  kReducePulse: sum (phi - phi_a)^2, sum phi_a^2;  kReduceField: same against
//  the field ref;  kReduceNonFinite: number of non-finite populations;  kReduceBadField: number of
//  values of ref that are not finite and > 0.
template <typename S, typename C, int KIND>
__device__ __forceinline__ void reduce_nodes(const S* P, const PlaneLayout& L, C phi_ref, const PulseTime& pt, double x0,
                                             double y0, double dx, const double* ref, double& a, double& b) {
    const unsigned stride = gridDim.x * blockDim.x, first = blockIdx.x * blockDim.x + threadIdx.x;
    auto against = [&](double phi, int i, int j) {
        const double r = KIND == kReducePulse ? pulse_phi(pt, x0 + i * dx, y0 + j * dx) : ref[(size_t)j * L.nx + i];
        const double d = phi - r;
        a += d * d;
        b += r * r;
    };
    if constexpr (KIND == kReduceBadField) {
        const unsigned n = (unsigned)L.nx * L.ny;
        unsigned bad = 0;
        for (unsigned k = first; k < n; k += stride) {
            const double v = ref[k];
            bad += (v > 0.0 && isfinite(v)) ? 0u : 1u;
        }
        a = (double)bad;
    } else if constexpr (sizeof(S) == 8) {
        const unsigned n = (unsigned)L.nx * L.ny;
        unsigned bad = 0;
        // four nodes' loads in flight (GB300, FP64 4096^2, us: the mass 370, now 352; against a field 418, now 410)
#pragma unroll 4
        for (unsigned k = first; k < n; k += stride) {
            const int j = (int)(k / L.nx), i = (int)(k - (unsigned)j * L.nx);
            if constexpr (KIND == kReduceNonFinite) {
#pragma unroll
                for (int q = 0; q < kQ; ++q) bad += isfinite(pulled<S, C>(P, q, i, j, L, phi_ref)) ? 0u : 1u;
            } else {
                const double phi = node_phi<S, C>(P, i, j, L, phi_ref);
                if constexpr (KIND == kReduceMass)
                    a += phi;
                else
                    against(phi, i, j);
            }
        }
        if constexpr (KIND == kReduceNonFinite) a = (double)bad;
    } else {
        const unsigned np = (L.nx + 1) / 2, n = np * L.ny;
        unsigned bad = 0;
        F2 s(0.f), c(0.f), t(0.f);  // mass: the thread's sum as s + c + t too
        for (unsigned k = first; k < n; k += stride) {
            const int j = (int)(k / np), i = 2 * (int)(k - (unsigned)j * np);
            const bool two = i + 1 < L.nx;
            if constexpr (KIND == kReduceNonFinite) {
                F2 g[kQ];
                pulled_pair(P, i, j, L, phi_ref, g);
#pragma unroll
                for (int q = 0; q < kQ; ++q) bad += (isfinite(g[q].v.x) ? 0u : 1u) + (two && !isfinite(g[q].v.y) ? 1u : 0u);
            } else {
                PhiPair p = pair_phi(P, i, j, L, phi_ref);
                if constexpr (KIND == kReduceMass) {
                    if (!float_sum_ok(p.s.v.x)) {
                        a += node_phi<S, C>(P, i, j, L, phi_ref);
                        p.s.v.x = p.c.v.x = p.t.v.x = 0.f;
                    }
                    if (!two || !float_sum_ok(p.s.v.y)) {
                        if (two) a += node_phi<S, C>(P, i + 1, j, L, phi_ref);
                        p.s.v.y = p.c.v.y = p.t.v.y = 0.f;
                    }
                    F2 e, f, g;
                    s = two_sum(s, p.s, e);
                    c = two_sum(c, p.c, f);
                    c = two_sum(c, e, g);
                    t = t + ((p.t + f) + g);
                    if (!(fabsf(s.v.x) < 1e36f && fabsf(s.v.y) < 1e36f)) {  // long before the float range ends
                        a += ((double)s.v.x + (double)s.v.y) + ((double)c.v.x + (double)c.v.y);
                        s = c = F2(0.f);
                    }
                } else {
                    against(phi_value(p.s.v.x, p.c.v.x, p.t.v.x, P, i, j, L, phi_ref), i, j);
                    if (two) against(phi_value(p.s.v.y, p.c.v.y, p.t.v.y, P, i + 1, j, L, phi_ref), i + 1, j);
                }
            }
        }
        if constexpr (KIND == kReduceNonFinite) a = (double)bad;
        if constexpr (KIND == kReduceMass)
            a += (((double)s.v.x + (double)s.v.y) + ((double)c.v.x + (double)c.v.y)) + ((double)t.v.x + (double)t.v.y);
    }
}

// Per-block FP64 partial sums into partial[2 * block + {0, 1}]; the last block to finish sums them in a
// fixed order into the pinned host result, beside the timeout flag.
template <typename S, typename C, int KIND>
__global__ void __launch_bounds__(kThreads)
    reduce_kernel(double* partial, unsigned* done, const S* P, PlaneLayout L, C phi_ref, PulseTime pt, double x0, double y0,
                  double dx, const double* ref, double* result, const int* flag, int* host_flag) {
    overlap_launch();
    __shared__ bool last;
    double a = 0.0, b = 0.0;
    reduce_nodes<S, C, KIND>(P, L, phi_ref, pt, x0, y0, dx, ref, a, b);
    block_sum2(a, b);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = a;
        partial[2 * blockIdx.x + 1] = b;
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    a = b = 0.0;
    for (unsigned k = threadIdx.x; k < gridDim.x; k += blockDim.x) {
        a += __ldcg(&partial[2 * k]);
        b += __ldcg(&partial[2 * k + 1]);
    }
    __syncthreads();  // block_sum2's shared arrays are used again
    block_sum2(a, b);
    if (threadIdx.x == 0) {
        result[0] = a;
        result[1] = b;
        *host_flag = *flag;
        *done = 0u;
    }
}

template <typename S, typename C>
__global__ void get_pop_kernel(double* g, const S* P, PlaneLayout L, C phi_ref, const int* flag, int* host_flag) {
    overlap_launch();
    report_flag(flag, host_flag);
    const unsigned n = (unsigned)L.nx * L.ny;
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int j = (int)(k / L.nx), i = (int)(k - (unsigned)j * L.nx);
#pragma unroll
        for (int q = 0; q < kQ; ++q) g[(size_t)q * n + k] = (double)pulled<S, C>(P, q, i, j, L, phi_ref);
    }
}

template <typename S, typename C>
__global__ void set_pop_kernel(S* P, const double* g, PlaneLayout L, C phi_ref) {
    overlap_launch();
    const unsigned n = (unsigned)L.nx * L.ny;
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int j = (int)(k / L.nx), i = (int)(k - (unsigned)j * L.nx);
        const bool inner = inner_node(L, i, j);
#pragma unroll
        for (int q = 0; q < kQ; ++q)
            store_pulled(P, L, q, i, j, inner, Store<S>::encode((C)g[(size_t)q * n + k], weight<C>(q) * phi_ref));
    }
}

template <typename S, typename C>
__global__ void sample_kernel(double* out, const long* nodes, int count, const S* P, PlaneLayout L, C phi_ref) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= count * kQ) return;
    const int s = t / kQ, q = t - s * kQ;
    const long k = nodes[s];
    const int j = (int)(k / L.nx), i = (int)(k - (long)j * L.nx);
    out[t] = (double)pulled<S, C>(P, q, i, j, L, phi_ref);
}

int grid_for(const trtr_ctx* ctx, size_t n) {
    const size_t want = (n + kThreads - 1) / kThreads;
    const size_t cap = (size_t)ctx->num_sms * 8;
    return (int)(want < 1 ? 1 : (want > cap ? cap : want));
}

// A launch that overlaps the tail of the kernel before it (overlap_launch).
template <typename... P, typename... A>
void launch_overlapped(trtr_ctx* ctx, void (*kernel)(P...), int grid, int threads, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// The pinned copy of the timeout flag.
int* host_flag(trtr_ctx* ctx) { return reinterpret_cast<int*>(ctx->hres + 3); }

template <typename F>
cudaError_t dispatch(trtr_ctx* ctx, F&& f) {
    switch (ctx->p.precision) {
        case TRTR_F64: f((double*)nullptr, (double*)nullptr); break;
        case TRTR_F32: f((float*)nullptr, (float*)nullptr); break;
        case TRTR_F16_OFS: f((__half*)nullptr, (float*)nullptr); break;
        case TRTR_BF16_OFS: f((__nv_bfloat16*)nullptr, (float*)nullptr); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_convert_fields(trtr_ctx* ctx, const double* ux, const double* uy, const double* D) {
    const size_t n = (size_t)(ctx->p.nx + 2) * (ctx->p.ny + 2);
    const double us = ctx->p.dt / ctx->p.dx, ds = ctx->p.dt / (ctx->p.dx * ctx->p.dx);
    const int use_const = ctx->p.tau1_const > 0.0;
    const double dh = use_const ? (ctx->p.tau1_const - 0.5) / 3.0 : 0.0;
    ctx->launches += 1;
    return dispatch(ctx, [&](auto* sp, auto* cp) {
        using C = std::remove_pointer_t<decltype(cp)>;
        (void)sp;
        convert_fields_kernel<C><<<grid_for(ctx, n), kThreads, 0, ctx->stream>>>(
            (C*)ctx->uv, (C*)ctx->Dh, ux, uy, D, ctx->lf, ctx->p.grad_mode, us, ds, dh, use_const);
    });
}

cudaError_t launch_pulse_fields(trtr_ctx* ctx) {
    const size_t n = (size_t)(ctx->p.nx + 2) * (ctx->p.ny + 2);
    const int use_const = ctx->p.tau1_const > 0.0;
    const double dh = use_const ? (ctx->p.tau1_const - 0.5) / 3.0 : 0.0;
    ctx->launches += 1;
    return dispatch(ctx, [&](auto* sp, auto* cp) {
        using C = std::remove_pointer_t<decltype(cp)>;
        (void)sp;
        pulse_fields_kernel<C><<<grid_for(ctx, n), kThreads, 0, ctx->stream>>>(
            (C*)ctx->uv, (C*)ctx->Dh, (C*)ctx->tab_x, (C*)ctx->tab_y, ctx->lf, ctx->p.grad_mode, ctx->p.x0, ctx->p.y0,
            ctx->p.dx, ctx->p.dt, ctx->pulse, dh, use_const);
    });
}

cudaError_t launch_convert_source(trtr_ctx* ctx, const double* S, int buffer) {
    const size_t n = (size_t)ctx->p.nx * ctx->p.ny;
    ctx->launches += 1;
    return dispatch(ctx, [&](auto* sp, auto* cp) {
        using C = std::remove_pointer_t<decltype(cp)>;
        (void)sp;
        launch_overlapped(ctx, convert_source_kernel<C>, grid_for(ctx, n), kThreads,
                          (C*)ctx->S + (size_t)buffer * ctx->lf.plane, S, ctx->lf, ctx->p.dt);
    });
}

cudaError_t launch_init_equilibrium(trtr_ctx* ctx, const double* phi0) {
    ctx->launches += 1;
    const int nx = ctx->p.nx, ny = ctx->p.ny;
    // the pulse: columns of a block, fewer where the last block of a row would leave more than a tenth of them
    // empty (GB300, us, 128 columns always / now: FP32 16 x 4000 26.9 / 8.0, 40 x 4000 24.9 / 10.5), and as many rows as
    // leave eight blocks an SM
    int log_w = 7;
    auto blocks = [&](int l) { return (nx + (1 << l) - 1) >> l; };
    while (log_w > 4 && 10L * (blocks(log_w) << log_w) > 11L * nx) --log_w;
    const int step = kInitThreads >> log_w, columns = blocks(log_w);
    const long share = (long)ny * columns / (8L * ctx->num_sms);
    const int rows = ((int)(share < 1 ? 1 : (share > kInitRows ? kInitRows : share)) + step - 1) / step * step;
    const PulseTime pt = pulse_at(ctx->pulse, 0.0);
    return dispatch(ctx, [&](auto* sp, auto* cp) {
        using S = std::remove_pointer_t<decltype(sp)>;
        using C = std::remove_pointer_t<decltype(cp)>;
        S* P = (S*)ctx->pop[ctx->cur];
        const C* uv = (const C*)ctx->uv;
        const C phi_ref = (C)ctx->p.phi_ref;
        if (phi0)
            init_eq_kernel<S, C><<<grid_for(ctx, (size_t)nx * ny), kThreads, 0, ctx->stream>>>(P, uv, phi0, ctx->lp, ctx->lf, phi_ref);
        else
            init_pulse_kernel<S, C><<<dim3(columns, (ny + rows - 1) / rows), kInitThreads, 0, ctx->stream>>>(
                P, uv, ctx->lp, ctx->lf, ctx->p.x0, ctx->p.y0, ctx->p.dx, pt, phi_ref, log_w, rows);
    });
}

cudaError_t launch_moments(trtr_ctx* ctx, double* phi_out) {
    const size_t n = (size_t)ctx->p.nx * ctx->p.ny;
    ctx->launches += 1;
    return dispatch(ctx, [&](auto* sp, auto* cp) {
        using S = std::remove_pointer_t<decltype(sp)>;
        using C = std::remove_pointer_t<decltype(cp)>;
        launch_overlapped(ctx, moments_kernel<S, C>, grid_for(ctx, sizeof(S) == 8 ? n : (n + 1) / 2), kThreads, phi_out,
                          (const S*)ctx->pop[ctx->cur], ctx->lp, (C)ctx->p.phi_ref, ctx->dflag, host_flag(ctx));
    });
}

template <int KIND>
cudaError_t launch_reduce_kind(trtr_ctx* ctx, const double* ref) {
    const PulseTime pt = pulse_at(ctx->pulse, (double)ctx->step * ctx->p.dt);
    ctx->launches += 1;
    return dispatch(ctx, [&](auto* sp, auto* cp) {
        using S = std::remove_pointer_t<decltype(sp)>;
        using C = std::remove_pointer_t<decltype(cp)>;
        launch_overlapped(ctx, reduce_kernel<S, C, KIND>, ctx->red_blocks, kThreads, ctx->scratch,
                          ctx->red_done, (const S*)ctx->pop[ctx->cur], ctx->lp,
                          (C)ctx->p.phi_ref, pt, ctx->p.x0, ctx->p.y0, ctx->p.dx, ref, ctx->hres, ctx->dflag, host_flag(ctx));
    });
}

cudaError_t launch_reduce(trtr_ctx* ctx, int kind, const double* ref) {
    switch (kind) {
        case kReduceMass: return launch_reduce_kind<kReduceMass>(ctx, ref);
        case kReducePulse: return launch_reduce_kind<kReducePulse>(ctx, ref);
        case kReduceField: return launch_reduce_kind<kReduceField>(ctx, ref);
        case kReduceNonFinite: return launch_reduce_kind<kReduceNonFinite>(ctx, ref);
        case kReduceBadField: return launch_reduce_kind<kReduceBadField>(ctx, ref);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_get_populations(trtr_ctx* ctx, double* g) {
    const size_t n = (size_t)ctx->p.nx * ctx->p.ny;
    ctx->launches += 1;
    return dispatch(ctx, [&](auto* sp, auto* cp) {
        using S = std::remove_pointer_t<decltype(sp)>;
        using C = std::remove_pointer_t<decltype(cp)>;
        launch_overlapped(ctx, get_pop_kernel<S, C>, grid_for(ctx, n), kThreads, g, (const S*)ctx->pop[ctx->cur], ctx->lp,
                          (C)ctx->p.phi_ref, ctx->dflag, host_flag(ctx));
    });
}

cudaError_t launch_set_populations(trtr_ctx* ctx, const double* g) {
    const size_t n = (size_t)ctx->p.nx * ctx->p.ny;
    ctx->launches += 1;
    return dispatch(ctx, [&](auto* sp, auto* cp) {
        using S = std::remove_pointer_t<decltype(sp)>;
        using C = std::remove_pointer_t<decltype(cp)>;
        launch_overlapped(ctx, set_pop_kernel<S, C>, grid_for(ctx, n), kThreads, (S*)ctx->pop[ctx->cur], g, ctx->lp,
                          (C)ctx->p.phi_ref);
    });
}

cudaError_t launch_sample(trtr_ctx* ctx, const long* nodes, int count, double* out) {
    ctx->launches += 1;
    const int total = count * kQ;
    return dispatch(ctx, [&](auto* sp, auto* cp) {
        using S = std::remove_pointer_t<decltype(sp)>;
        using C = std::remove_pointer_t<decltype(cp)>;
        sample_kernel<S, C><<<(total + kThreads - 1) / kThreads, kThreads, 0, ctx->stream>>>(
            out, nodes, count, (const S*)ctx->pop[ctx->cur], ctx->lp, (C)ctx->p.phi_ref);
    });
}

cudaError_t launch_gather_edges(trtr_ctx* ctx, const double* phi_b) {
    const int nb = edge_count(ctx->p.nx, ctx->p.ny);
    ctx->launches += 1;
    launch_overlapped(ctx, gather_edges_kernel, (nb + 31) / 32, 32, ctx->phib, phi_b, ctx->p.nx, ctx->p.ny);
    return cudaGetLastError();
}

cudaError_t launch_dirichlet(trtr_ctx* ctx, void* P) {
    const int nb = edge_count(ctx->p.nx, ctx->p.ny);
    ctx->launches += 1;
    return dispatch(ctx, [&](auto* sp, auto* cp) {
        using S = std::remove_pointer_t<decltype(sp)>;
        using C = std::remove_pointer_t<decltype(cp)>;
        launch_overlapped(ctx, dirichlet_nee_kernel<S, C>, (kQ * nb + 31) / 32, 32, (S*)P, (const C*)ctx->uv, ctx->phib,
                          ctx->lp, ctx->lf, (C)ctx->p.phi_ref);
    });
}

TRTR_BOUNDS_TAKE(aux)

}  // namespace trtr
