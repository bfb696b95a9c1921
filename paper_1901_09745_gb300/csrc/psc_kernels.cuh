// psc_kernels.cuh -- sm_103a kernels of one lattice-Boltzmann step with the modified
// partially-saturated-cell (PSC) immersed moving boundary (Liu & Wu, arXiv 1901.09745).
//
// The lattice is cut into tiles of 256 cells (tile_ext). After binning, k_pack_tiles writes each
// tile's candidate particles as packed records and sorts the tiles into three lists: tiles
// without candidates, tiles with at most 32 (both by k_step in psc_pair.cuh, 16-bit storage by
// the kernels of psc_pair16.cuh), tiles with more (the exact chunked path of k_collide_overflow,
// psc_tile below). Per cell every path
//   1. pulls the Q post-collision populations of the previous step from the neighbours
//      x - e_i (Eq. 1; periodic wrap; halfway bounce-back at walls, Eq. 6),
//   2. forms rho and the force-shifted u (Eq. 5),
//   3. walks the tile's candidate particles and computes each particle's solid fraction by the
//      linear approximation (Eq. 15-18, Table 1),
//   4. forms eps_n, B_n (Eq. 9) and the per-particle weights B_{n,s} (Eq. 13),
//   5. collides with BGK + Guo forcing + sum_s B_{n,s} Omega^s (Eq. 2-4, 10, 12) and
//      stores the Q post-collision populations of its own cell,
//   6. reduces each particle's momentum exchange B_{n,s} sum_i Omega^s_i e_i and its
//      torque (Eq. 14) over the warp with shuffles (16 bits and psc_tile: then over the block)
//      and adds the total with one FP64 atomic per particle and component.
//
// Two algebraic identities keep the per-candidate work independent of Q (exact up to
// rounding order, derived from Eq. 3 and Eq. 10):
//   sum_s B_{n,s} f_i^eq(rho, u_s) = rho w_i [B_n + 3 e_i.m + 9/2 e_i.M.e_i - 3/2 tr M],
//       m = sum_s B_{n,s} u_s, M = sum_s B_{n,s} u_s u_s^T   (f^eq is quadratic in u_s);
//   sum_i Omega^s_i e_i = rho (u + u_s) - 2 j = rho u_s + F/2 - j,   j = sum_i f_i e_i.
// Populations are stored as deviations d_i = f_i - w_i, so every stored and summed value
// is small and FP32 keeps its relative precision (rho = 1 + sum_i d_i).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lattice.cuh"
#include "hostdev.cuh"
#include "psc_internal.h"

namespace psc {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr unsigned kFull = 0xffffffffu;

template <typename T> struct PhysT {
    T omega;        // 1/tau
    T tmh;          // tau - 1/2
    T guo;          // 1 - 1/(2 tau), Eq. 4
    T F[3];         // body force
    T h;            // Table 1 shell half-width
    float2 sc;      // (scale, 1/scale) of the stored deviations
    T none;         // 0, unknown to the compiler
    T c12[2];       // 1 / 12 in the compute type and what that rounding left
    int inax;       // axis whose low face is an inlet (-1: none)
    T inua;         // inlet velocity along that axis
    T ineu[19];     // 6 w_i (e_i . u_in): f^eq_i - f^eq_{-i} of Eq. 3 at rho = 1
};

template <typename T> __host__ PhysT<T> make_phys(const Phys &ph, const int lattice = 19) {
    PhysT<T> k;
    k.omega = (T)(1.0 / ph.tau);
    k.tmh = (T)(ph.tau - 0.5);
    k.guo = (T)(1.0 - 1.0 / (2.0 * ph.tau));
    for (int a = 0; a < 3; ++a) k.F[a] = (T)ph.body_force[a];
    k.h = (T)ph.shell_h;
    k.sc = make_float2((float)ph.scale, (float)(1.0 / ph.scale));
    k.none = (T)0;
    k.c12[0] = (T)(1.0 / 12.0);
    k.c12[1] = (T)(1.0 / 12.0 - (double)k.c12[0]);
    const double *u = ph.inflow;
    k.inax = ph.inflow_axis;
    k.inua = (T)(ph.inflow_axis >= 0 ? u[ph.inflow_axis] : 0.0);   // the inlet is a low face
    for (int i = 0; i < 19; ++i) {
        double eu = 0.0, w = 0.0;
        if (lattice == 9 && i < 9) { eu = D2Q9::ex(i) * u[0] + D2Q9::ey(i) * u[1]; w = weight<D2Q9>(i); }
        else if (lattice == 19) { eu = D3Q19::ex(i) * u[0] + D3Q19::ey(i) * u[1] + D3Q19::ez(i) * u[2]; w = weight<D3Q19>(i); }
        k.ineu[i] = (T)(6.0 * w * eu);
    }
    return k;
}

// Velocity inlet (reading of Sec. 3.2's "constant flow with velocity U0"): on the inlet face
// the populations coming in (e_a = +1 along the inlet axis a) are not known from a
// neighbour; they take the non-equilibrium part of the opposite population, f_i = f_{-i} +
// f^eq_i(rho, u_in) - f^eq_{-i}(rho, u_in) = f_{-i} + 6 w_i rho e_i.u_in, with the density that
// gives the face cell the velocity u_in along a: rho (1 - u_a) = sum_{e_a = 0} f + 2 sum_{e_a = -1} f.
// df holds deviations (scaled by s when RAW); the directions in `fill` (those whose source
// lies beyond the inlet and beyond no wall) are overwritten.
template <class L, bool RAW, typename T>
__device__ __forceinline__ void inflow_nebb(T *df, const PhysT<T> &ph, const float2 sc, const unsigned fill) {
    const int a = ph.inax;
    T sd = (T)0;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const int ea = (a == 0) ? L::ex(i) : ((a == 1) ? L::ey(i) : L::ez(i));
        if (ea == 0) sd += df[i];
        else if (ea == -1) sd += (T)2 * df[i];
    }
    const T s = RAW ? (T)sc.x : (T)1;
    // sum_{e_a = 0} w + 2 sum_{e_a = -1} w = 1, so the deviations give rho directly
    const T rho = ((T)1 + sd / s) / ((T)1 - ph.inua);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        if (fill & (1u << i)) df[i] = df[opp<L>(i)] + s * rho * ph.ineu[i];
    }
}

// Constant-pressure outlet (reading of Sec. 3.2's outlet), on the high face of the inlet axis
// a: the populations coming in (e_a = -1) are unknown; the density is held at 1 and the
// velocity across the face follows from the known ones, 1 + u_a = sum_{e_a = 0} f +
// 2 sum_{e_a = +1} f; the unknown ones are f_i = f_{-i} + 6 w_i e_{i,a} u_a (the difference of
// the equilibria of Eq. 3 at rho = 1, u = u_a along a).
template <class L, bool RAW, typename T>
__device__ __forceinline__ void outlet_nebb(T *df, const PhysT<T> &ph, const float2 sc, const unsigned fill) {
    const int a = ph.inax;
    T sd = (T)0;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const int ea = (a == 0) ? L::ex(i) : ((a == 1) ? L::ey(i) : L::ez(i));
        if (ea == 0) sd += df[i];
        else if (ea == 1) sd += (T)2 * df[i];
    }
    // sum_{e_a = 0} w + 2 sum_{e_a = +1} w = 1: the scaled deviation sum is s u_a
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const int ea = (a == 0) ? L::ex(i) : ((a == 1) ? L::ey(i) : L::ez(i));
        if (fill & (1u << i)) df[i] = df[opp<L>(i)] + (T)(6.0 * weight<L>(i)) * (T)ea * sd;
    }
    (void)sc;
}

// Programmatic dependent launch within the step: a kernel launched with launch_pdl may start
// while its predecessor in the stream finishes; it calls pdl_wait() before it reads anything
// the predecessor wrote, and pdl_launch() lets its own successor start early.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// Is cell (x, y, z) one this context updates (inside the lattice and, in a slab of a
// decomposed lattice, outside its ghost layers along the slowest axis; act1 <= n there)?
template <class L>
__device__ __forceinline__ bool cell_active(const Geom &g, const int x, const int y, const int z) {
    if (L::D == 2) return x < g.n[0] && (unsigned)(y - g.act0) < (unsigned)(g.act1 - g.act0);
    return x < g.n[0] && y < g.n[1] && (unsigned)(z - g.act0) < (unsigned)(g.act1 - g.act0);
}

__device__ __forceinline__ float  rint_t(float v) { return rintf(v); }
__device__ __forceinline__ double rint_t(double v) { return rint(v); }
__device__ __forceinline__ float  sqrt_t(float v) { return sqrtf(v); }
__device__ __forceinline__ double sqrt_t(double v) { return sqrt(v); }
// Distances of cells from particle centres in the solid-fraction and row tests: FP32 takes
// v * rsqrt(v) (a few ulp, far below the FP32 parity tolerance; two instructions instead of
// the correctly rounded square root); FP64 keeps the correctly rounded one.
__device__ __forceinline__ float  dist_t(float v) { return v > 0.0f ? v * rsqrtf(v) : 0.0f; }
__device__ __forceinline__ double dist_t(double v) { return sqrt(v); }

// Population i of cell (x, y, z) after streaming: the value the neighbour x - e_i stored
// in the previous step, or, when x - e_i lies beyond a wall, the value this cell stored in
// the opposite direction (halfway bounce-back, Eq. 6). Periodic and wall faces only.
template <class L, typename S>
__device__ __forceinline__ typename Store<S>::T
pull_one(const S *__restrict__ fin, const Geom &g, int x, int y, int z, long long cell, int i,
         float2 sc) {
    int s[3] = {x - L::ex(i), y - L::ey(i), z - L::ez(i)};
    bool bounce = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (s[a] < 0 || s[a] >= g.n[a]) {
            if (g.periodic[a]) s[a] += (s[a] < 0) ? g.n[a] : -g.n[a];
            else bounce = true;
        }
    }
    if (bounce) return Store<S>::ld(fin, PSC_IDX((long long)opp<L>(i) * g.ncell + cell, L::Q * g.ncell, CHK_POP), sc);
    long long src = (long long)s[0] + (long long)g.n[0] * ((long long)s[1] + (long long)g.n[1] * s[2]);
    return Store<S>::ld(fin, PSC_IDX((long long)i * g.ncell + src, L::Q * g.ncell, CHK_POP), sc);
}

// The same for every face kind: beyond an open face the source is clamped onto the face
// (zero gradient); beyond the inlet or the outlet face the population is unknown (returned
// as 0, `from_inlet` or `from_outlet` set) and is filled in by inflow_nebb or outlet_nebb
// once all are pulled. A wall takes precedence over the inlet and outlet faces, these over
// open faces.
template <class L, typename S>
__device__ __forceinline__ typename Store<S>::T
pull_one_faces(const S *__restrict__ fin, const Geom &g, int x, int y, int z, long long cell, int i,
               float2 sc, bool &from_inlet, bool &from_outlet) {
    int s[3] = {x - L::ex(i), y - L::ey(i), z - L::ez(i)};
    bool bounce = false, inflow = false, outflow = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (s[a] < 0 || s[a] >= g.n[a]) {
            const int kind = face_kind(g, a, s[a] < 0 ? 0 : 1);
            if (kind == FACE_PERIODIC) s[a] += (s[a] < 0) ? g.n[a] : -g.n[a];
            else if (kind == FACE_WALL) bounce = true;
            else if (kind == FACE_OPEN) s[a] = (s[a] < 0) ? 0 : g.n[a] - 1;
            else if (kind == FACE_INFLOW) inflow = true;
            else outflow = true;
        }
    }
    if (bounce) return Store<S>::ld(fin, PSC_IDX((long long)opp<L>(i) * g.ncell + cell, L::Q * g.ncell, CHK_POP), sc);
    from_inlet = inflow;
    from_outlet = outflow && !inflow;
    if (inflow || outflow) return (typename Store<S>::T)0;
    long long src = (long long)s[0] + (long long)g.n[0] * ((long long)s[1] + (long long)g.n[1] * s[2]);
    return Store<S>::ld(fin, PSC_IDX((long long)i * g.ncell + src, L::Q * g.ncell, CHK_POP), sc);
}

// All Q populations of cell (x, y, z) after streaming, one pull_one per direction, the
// unknown ones at an inlet filled in.
template <class L, typename S>
__device__ __forceinline__ void pull_all(const S *__restrict__ fin, const Geom &g, int x, int y, int z,
                                         long long cell, const PhysT<typename Store<S>::T> &ph,
                                         typename Store<S>::T *df) {
    unsigned fill = 0u, fillo = 0u;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        bool in = false, out = false;
        df[i] = pull_one_faces<L, S>(fin, g, x, y, z, cell, i, ph.sc, in, out);
        if (in) fill |= 1u << i;
        if (out) fillo |= 1u << i;
    }
    if (fill) inflow_nebb<L, false>(df, ph, ph.sc, fill);
    if (fillo) outlet_nebb<L, false>(df, ph, ph.sc, fillo);
}

// Warp sum of NV values per lane (NV a power of two <= 32) in NV - 1 + 5 - log2(NV) shuffles
// instead of 5 NV: each butterfly stage first halves the set of values a lane carries (it
// keeps one half and sends the other to its partner), then plain butterflies finish. On
// return lane l holds the warp total of value l >> (5 - log2 NV).
template <int NV, typename T>
__device__ __forceinline__ T warp_sum_spread(T (&v)[NV], const int lane) {
    int m = NV;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        if (m > 1) {
            const int half = m >> 1;
            const bool up = (lane & off) != 0;
#pragma unroll
            for (int j = 0; j < NV / 2; ++j) {
                if (j < half) {
                    const T snd = up ? v[j] : v[j + half];
                    const T kp = up ? v[j + half] : v[j];
                    v[j] = kp + __shfl_xor_sync(kFull, snd, off);
                }
            }
            m = half;
        } else {
            v[0] += __shfl_xor_sync(kFull, v[0], off);
        }
    }
    return v[0];
}

// e_i . v for a lattice velocity with components in {-1, 0, 1}: additions only, no
// multiplications by 0 or 1 (which IEEE arithmetic does not let the compiler drop).
template <class L, typename T>
__device__ __forceinline__ T edot(const int i, const T vx, const T vy, const T vz) {
    const int ex = L::ex(i), ey = L::ey(i), ez = L::ez(i);
    T r = (T)0;
    bool first = true;
    if (ex) { r = ex > 0 ? vx : -vx; first = false; }
    if (ey) { r = first ? (ey > 0 ? vy : -vy) : (ey > 0 ? r + vy : r - vy); first = false; }
    if (ez) { r = first ? (ez > 0 ? vz : -vz) : (ez > 0 ? r + vz : r - vz); }
    return r;
}

// Where the pull of direction i at cell x reads (Eq. 1, 6): x - e_i, or the cell itself in
// direction -i when x - e_i lies beyond a wall (halfway bounce-back). The offsets to the -1
// and +1 neighbour on each axis (periodic wrap folded in) and the wall flags are formed once
// per cell, so each direction costs an add and a select instead of three range tests. The
// adjoint pushes to the same index.
struct NbrIdx {
    long long oxm, oxp, oym, oyp, ozm, ozp;   // source offsets when e = +1 (m) / -1 (p)
    unsigned wall;                            // bits 0..5: wxm wxp wym wyp wzm wzp
};

template <class L>
__device__ __forceinline__ NbrIdx make_nbr_idx(const Geom &g, int x, int y, int z) {
    const long long sy = g.n[0], sz = (long long)g.n[0] * g.n[1];
    NbrIdx nb{-1, 1, -sy, sy, -sz, sz, 0u};
    if (x == 0) { if (g.periodic[0]) nb.oxm = g.n[0] - 1; else nb.wall |= 1u; }
    if (x == g.n[0] - 1) { if (g.periodic[0]) nb.oxp = -(long long)(g.n[0] - 1); else nb.wall |= 2u; }
    if (y == 0) { if (g.periodic[1]) nb.oym = (long long)(g.n[1] - 1) * sy; else nb.wall |= 4u; }
    if (y == g.n[1] - 1) { if (g.periodic[1]) nb.oyp = -(long long)(g.n[1] - 1) * sy; else nb.wall |= 8u; }
    if (L::D == 3) {
        if (z == 0) { if (g.periodic[2]) nb.ozm = (long long)(g.n[2] - 1) * sz; else nb.wall |= 16u; }
        if (z == g.n[2] - 1) { if (g.periodic[2]) nb.ozp = -(long long)(g.n[2] - 1) * sz; else nb.wall |= 32u; }
    }
    return nb;
}

template <class L>
__device__ __forceinline__ long long src_index(const NbrIdx &nb, const int i, const long long cell, const long long N) {
    long long off = 0;
    unsigned w = 0u;
    if (L::ex(i) == 1) { off += nb.oxm; w |= 1u; }
    if (L::ex(i) == -1) { off += nb.oxp; w |= 2u; }
    if (L::ey(i) == 1) { off += nb.oym; w |= 4u; }
    if (L::ey(i) == -1) { off += nb.oyp; w |= 8u; }
    if (L::ez(i) == 1) { off += nb.ozm; w |= 16u; }
    if (L::ez(i) == -1) { off += nb.ozp; w |= 32u; }
    return (nb.wall & w) ? (long long)opp<L>(i) * N + cell : (long long)i * N + cell + off;
}

// All Q pulled deviations of the cell (x, y, z). Tiles one cell clear of every face use
// fixed offsets; elsewhere the same offsets and wall flags as make_nbr_idx, held in scalars
// (measured faster here than going through the struct).
template <class L, typename S, bool RAW = false>
__device__ __forceinline__ void pull_q(const S *__restrict__ fin, const Geom &g, int x, int y, int z,
                                       long long cell, bool interior, bool active, float2 sc,
                                       typename Store<S>::T *df) {
    constexpr int Q = L::Q;
    using T = typename Store<S>::T;
    const long long N = g.ncell;
    const long long sy = g.n[0], sz = (long long)g.n[0] * g.n[1];
    if (interior) {
        const S *base = fin + cell;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const long long o = (long long)i * N - (L::ex(i) + L::ey(i) * sy + L::ez(i) * sz);
            const long long oc = PSC_OFF(cell, o, Q * N, CHK_POP);
            df[i] = RAW ? Store<S>::ldr(base, oc) : Store<S>::ld(base, oc, sc);
        }
        return;
    }
    if (!active) {
#pragma unroll
        for (int i = 0; i < Q; ++i) df[i] = (T)0;
        return;
    }
    // source x - e: from the -1 neighbour when e = +1 (m), from the +1 neighbour when e = -1 (p);
    // periodic and wall faces only (contexts with open, inlet or outlet faces step with
    // k_collide_faces)
    long long oxm = -1, oxp = 1, oym = -sy, oyp = sy, ozm = -sz, ozp = sz;
    bool wxm = false, wxp = false, wym = false, wyp = false, wzm = false, wzp = false;
    if (x == 0) { if (g.periodic[0]) oxm = g.n[0] - 1; else wxm = true; }
    if (x == g.n[0] - 1) { if (g.periodic[0]) oxp = -(long long)(g.n[0] - 1); else wxp = true; }
    if (y == 0) { if (g.periodic[1]) oym = (long long)(g.n[1] - 1) * sy; else wym = true; }
    if (y == g.n[1] - 1) { if (g.periodic[1]) oyp = -(long long)(g.n[1] - 1) * sy; else wyp = true; }
    if (L::D == 3) {
        if (z == 0) { if (g.periodic[2]) ozm = (long long)(g.n[2] - 1) * sz; else wzm = true; }
        if (z == g.n[2] - 1) { if (g.periodic[2]) ozp = -(long long)(g.n[2] - 1) * sz; else wzp = true; }
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        long long off = 0;
        bool wall = false;
        if (L::ex(i) == 1) { off += oxm; wall |= wxm; }
        if (L::ex(i) == -1) { off += oxp; wall |= wxp; }
        if (L::ey(i) == 1) { off += oym; wall |= wym; }
        if (L::ey(i) == -1) { off += oyp; wall |= wyp; }
        if (L::ez(i) == 1) { off += ozm; wall |= wzm; }
        if (L::ez(i) == -1) { off += ozp; wall |= wzp; }
        const long long idx = wall ? (long long)opp<L>(i) * N + cell : (long long)i * N + cell + off;
        const long long ic = PSC_IDX(idx, Q * N, CHK_POP);
        df[i] = RAW ? Store<S>::ldr(fin, ic) : Store<S>::ld(fin, ic, sc);
    }
}

// ------------------------------------------------------------------- candidate records
// Each lattice tile owns one block of candidate records in global memory, written by the
// packing kernel after binning: a 16-byte header whose first element is the tile's
// candidate count, then up to `cap` records of RW values of the compute type, sorted by
// particle index (so per-cell sums do not depend on the binning's atomic order). A record
// holds the particle's position relative to the tile origin (minimum image; in wide tiles
// to its middle along x), radius, f(r) of Eq. 18 (negative for a particle that moves or
// spins), velocity, spin and index.
constexpr int RW = 12;
enum { R_PX = 0, R_PY, R_PZ, R_R, R_FR, R_UX, R_UY, R_UZ, R_OX, R_OY, R_OZ, R_ID };

template <typename T> __host__ __device__ constexpr int head_elems() { return 16 / (int)sizeof(T); }
template <typename T> __host__ __device__ inline long long block_elems(int cap) {
    return ((head_elems<T>() + (long long)cap * RW + 3) / 4) * 4;
}
template <typename T> __host__ __device__ inline size_t cs_smem_bytes(int cap, int nc) {
    return (size_t)cap * RW * sizeof(T) + (size_t)kWarps * cap * nc * sizeof(T);
}

// Particle index stored in a record slot as raw bits (no conversion instruction).
template <typename T> __device__ __forceinline__ T id_bits(int id);
template <> __device__ __forceinline__ float id_bits<float>(int id) { return __int_as_float(id); }
template <> __device__ __forceinline__ double id_bits<double>(int id) { return __longlong_as_double((long long)id); }
__device__ __forceinline__ int bits_id(float v) { return __float_as_int(v); }
__device__ __forceinline__ int bits_id(double v) { return (int)__double_as_longlong(v); }

// Record of particle `id` for the tile with origin (x0, y0, z0).
template <class L, typename T>
__device__ __forceinline__ void write_record(T *rec, const Geom &g, const Parts &pd, int id, int x0,
                                             int y0, int z0) {
    const int org[3] = {x0, y0, z0};
    const int ext[3] = {L::TX, L::TY, L::TZ};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        T rel = (T)0;
        if (a < L::D) {
            // minimum image with respect to the tile centre, one exact FP64 subtraction
            rel = (T)(record_rel(pd.X[3 * id + a], org[a], ext[a], g.n[a], g.inv_n[a], g.periodic[a]) - (a == 0 ? L::REC_X : 0));
        }
        rec[R_PX + a] = rel;
    }
    if (sizeof(T) == 4 && pd.Pf) {   // FP32 records: the per-particle copy, no conversions here
        const float4 a = pd.Pf[2 * id], b = pd.Pf[2 * id + 1];
        rec[R_R] = (T)a.x; rec[R_FR] = (T)a.y;
        rec[R_UX] = (T)a.z; rec[R_UY] = (T)a.w; rec[R_UZ] = (T)b.x;
        rec[R_OX] = (T)b.y; rec[R_OY] = (T)b.z; rec[R_OZ] = (T)b.w;
    } else {
        rec[R_R] = (T)pd.R[id];
        rec[R_FR] = (T)pd.Fr[id];
        rec[R_UX] = (T)pd.U[3 * id + 0]; rec[R_UY] = (T)pd.U[3 * id + 1]; rec[R_UZ] = (T)pd.U[3 * id + 2];
        rec[R_OX] = (T)pd.Om[3 * id + 0]; rec[R_OY] = (T)pd.Om[3 * id + 1]; rec[R_OZ] = (T)pd.Om[3 * id + 2];
    }
    // f(r) > 0: a negative one marks a particle that moves or spins
    bool moves = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) moves |= (rec[R_UX + a] != (T)0) || (rec[R_OX + a] != (T)0);
    if (moves) rec[R_FR] = -rec[R_FR];
    rec[R_ID] = id_bits<T>(id);
}

// Packing kernel: one warp per tile sorts the tile's candidate list and writes its block.
// Each block of 8 tiles then appends its tiles to the list of tiles with candidates or to
// the list of tiles without, and tiles with more candidates than `cap` also to the overflow
// list (tiles with more than min(cap, kPairCap) candidates; one atomic per list and block), so
// the collide-stream kernels run over compact lists and launch no block for a tile that is
// not theirs.
template <class L, typename T>
__global__ void k_pack_tiles(Geom g, Tiles tl, Parts pd, long long ntiles) {
    __shared__ int s_id[kWarps][64];
    __shared__ int s_cnt[kWarps];
    pdl_wait();       // the binning kernel's counts and lists
    pdl_launch();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // grid (nt0 / 8 * nt1, 1, nt2): the block's 8 warps take 8 tiles along x
    const unsigned nbx = (unsigned)(g.nt[0] + kWarps - 1) / kWarps, by = blockIdx.x / nbx;
    const int tx = (int)(blockIdx.x - by * nbx) * kWarps + warp, ty = (int)by, tz = (int)blockIdx.z;
    const long long tile = tx + (long long)g.nt[0] * (ty + (long long)g.nt[1] * tz);
    const bool valid = tx < g.nt[0];
    const int cnt = valid ? tl.count[tile] : -1;
    if (lane == 0) s_cnt[warp] = cnt;
    __syncthreads();
    // the lists first: their atomics are under way while the records are written
    if (warp == 0) {
        const int c = lane < kWarps ? s_cnt[lane] : -1, lim = min(tl.cap, kPairCap);
        const unsigned mp = __ballot_sync(kFull, c > 0), mf = __ballot_sync(kFull, c == 0), mo = __ballot_sync(kFull, c > lim);
        const unsigned mine = lane == 0 ? mp : (lane == 1 ? mf : (lane == 2 ? mo : 0u));
        const int at = mine ? atomicAdd(&tl.stats[lane == 0 ? 4 : (lane == 1 ? 5 : 2)], __popc(mine)) : 0;
        const int bp = __shfl_sync(kFull, at, 0), bf = __shfl_sync(kFull, at, 1), bo = __shfl_sync(kFull, at, 2);
        const unsigned below = (1u << lane) - 1u, ent = (unsigned)(tile + lane);      // the first warp's tile + lane
        if (c > 0) tl.order[bp + __popc(mp & below)] = ent;
        else if (c == 0) tl.order[ntiles + bf + __popc(mf & below)] = ent;
        if (c > lim) tl.order[2 * ntiles + bo + __popc(mo & below)] = ent;
    }
    if (valid) {
        const int m = min(cnt, tl.cap);
        T *blk = reinterpret_cast<T *>(tl.blocks) + tile * block_elems<T>(tl.cap);
        if (lane == 0) blk[0] = (T)cnt;
        for (int k = lane; k < m; k += 32) s_id[warp][k] = tl.list[tile * tl.cap + k];
        __syncwarp();
        for (int k = lane; k < m; k += 32) {
            const int id = (int)PSC_IDX(s_id[warp][k], pd.n, CHK_PART);
            int rank = 0;
            for (int q = 0; q < m; ++q) rank += (s_id[warp][q] < id);
            write_record<L, T>(blk + head_elems<T>() + (long long)rank * RW, g, pd, id, tx * L::TX, ty * L::TY,
                               tz * L::TZ);
        }
    }
}

// The geometric part of a record (position, radius) and the rest (f(r), U, Omega, index),
// read from shared memory with 16-byte loads (records are 16-byte aligned).
template <typename T> struct Vec4 { T x, y, z, w; };
template <typename T> __device__ __forceinline__ Vec4<T> ld4(const T *p);
template <> __device__ __forceinline__ Vec4<float> ld4<float>(const float *p) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    return {v.x, v.y, v.z, v.w};
}
template <> __device__ __forceinline__ Vec4<double> ld4<double>(const double *p) {
    const double2 a = *reinterpret_cast<const double2 *>(p);
    const double2 b = *reinterpret_cast<const double2 *>(p + 2);
    return {a.x, a.y, b.x, b.y};
}

// Arm x_n - X_p from the cell (cx, cy, cz) to the candidate at (px, py, pz), all relative
// to the tile origin, with the per-cell minimum image on short periodic axes.
template <class L, typename T>
__device__ __forceinline__ void cand_arm(const Geom &g, T cx, T cy, T cz, T px, T py, T pz, T &dx, T &dy,
                                         T &dz) {
    dx = cx - px;
    dy = cy - py;
    dz = (L::D == 3) ? cz - pz : (T)0;
    if (g.wrap_img[0]) dx -= (T)g.n[0] * rint_t(dx / (T)g.n[0]);
    if (g.wrap_img[1]) dy -= (T)g.n[1] * rint_t(dy / (T)g.n[1]);
    if (L::D == 3 && g.wrap_img[2]) dz -= (T)g.n[2] * rint_t(dz / (T)g.n[2]);
}

// Table 1 Steps 2-4 for a cell at squared distance d2 from a candidate of radius r:
// distance <= r - h -> 1, >= r + h -> 0, else clamp(f(r) - D, 0, 1) with D = distance - r.
template <typename T>
__device__ __forceinline__ T shell_eps(T d2, T r, T fr, T h) {
    fr = fabs(fr);      // a record marks moving particles by the sign
    const T rh = r + h;
    if (!(d2 < rh * rh)) return (T)0;
    const T ri = r - h;
    if (ri > (T)0 && d2 <= ri * ri) return (T)1;
    const T dist = dist_t(d2);
    if (dist <= ri) return (T)1;
    T e = fr - (dist - r);
    e = e < (T)0 ? (T)0 : e;
    e = e > (T)1 ? (T)1 : e;
    return e;
}

// Can the candidate at (px, py, pz) with reach R = r + h touch any cell of this warp's row
// (tile-relative y = cy, z = cz, x = 0..xmax)? Conservative: a false "yes" only costs time.
template <class L, typename T>
__device__ __forceinline__ bool row_hits(const Geom &g, T px, T py, T pz, T R, T cy, T cz, T xmax) {
    T dx, dy, dz;
    cand_arm<L, T>(g, (T)0, cy, cz, (T)0, py, pz, dx, dy, dz);
    const T rem = R * R - dy * dy - dz * dz;
    if (!(rem > (T)0)) return false;
    if (g.wrap_img[0]) return true;
    const T hw = dist_t(rem);
    return (px - hw <= xmax + (T)1) && (px + hw >= (T)-1);
}

// Tiles with candidate particles. The tile's records are staged in shared memory while the
// population loads are in flight. Each warp is one row of the tile: it culls the candidates
// that cannot reach its row (one lane per candidate, ballot), then every lane evaluates the
// remaining ones from shared memory (broadcast reads). Warps with no solid cell run the plain
// BGK + Guo update. Forces: each warp reduces each of its candidates' momentum exchange with
// shuffles; partial sums meet in shared memory and are added in a fixed order, one FP64
// atomic per particle and component per tile. Tiles with more candidates than the block
// holds take the same path chunk by chunk over all particles (exact, slow, rare).
template <class L, typename S, int PSC, bool FACES = false, bool FLUID = false>
__device__ __forceinline__ void psc_tile(const unsigned tile, const S *__restrict__ fin, S *__restrict__ fout,
                                         const Geom &g, const PhysT<typename Store<S>::T> &ph, const Tiles &tl,
                                         const Parts &pd, int *flags, typename Store<S>::T *srec,
                                         unsigned long long *s_mask) {
    using T = typename Store<S>::T;
    constexpr int Q = L::Q;
    constexpr int NC = (L::D == 2) ? 3 : 6;
    constexpr int NSLOT = 4;
    const int cap = tl.cap;
    T *part = srec + (size_t)cap * RW;                     // [kWarps][cap][NC] warp partials

    // (FLUID: a tile without candidates)
    const int cnt = FLUID ? 0 : tl.count[tile];
    const unsigned txy = tile / (unsigned)g.nt[0];          // 32-bit: tiles < 2^31 (host check)
    const int tx = (int)(tile - txy * (unsigned)g.nt[0]);
    const int ty = (int)(txy % (unsigned)g.nt[1]);
    const int tz = (int)(txy / (unsigned)g.nt[1]);
    const bool ovf = cnt > cap;
    const int nchunk = ovf ? (pd.n + cap - 1) / cap : 1;
    const T *recs = FLUID ? nullptr
                  : reinterpret_cast<const T *>(tl.blocks) + (size_t)tile * block_elems<T>(cap) + head_elems<T>();

    const int tid = threadIdx.x + L::TX * (threadIdx.y + L::TY * threadIdx.z);
    const int lane = tid & 31, warp = tid >> 5;
    const int x0 = tx * L::TX, y0 = ty * L::TY, z0 = tz * L::TZ;
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y, z = z0 + threadIdx.z;
    const bool active = cell_active<L>(g, x, y, z);
    const long long cell = x + (long long)g.n[0] * (y + (long long)g.n[1] * z);
    const long long N = g.ncell;

    // ---- 0. this thread's share of the tile's records (cap <= 64 records of RW values),
    //         loaded now, written to shared memory once the pull loads are in flight
    constexpr int kRecWords = (64 * RW + kThreads - 1) / kThreads;
    T rw[kRecWords];
    const int nwords = ovf ? 0 : cnt * RW;
#pragma unroll
    for (int j = 0; j < kRecWords; ++j) {
        const int w = tid + j * kThreads;
        rw[j] = (w < nwords) ? recs[w] : (T)0;
    }

    // ---- 1. pull (Eq. 1, Eq. 6)
    T df[Q];
    const bool interior = x0 >= 1 && x0 + L::TX < g.n[0] && y0 >= 1 && y0 + L::TY < g.n[1] &&
                          (L::D == 2 || (z0 >= 1 && z0 + L::TZ < g.n[2]));
    if (interior) {
        const S *base = fin + cell;
        const long long sy = g.n[0], sz = (long long)g.n[0] * g.n[1];
#pragma unroll
        for (int i = 0; i < Q; ++i)
            df[i] = Store<S>::ld(base, PSC_OFF(cell, (long long)i * N - (L::ex(i) + L::ey(i) * sy + L::ez(i) * sz), Q * N, CHK_POP), ph.sc);
    } else if (active) {
        if (FACES) {
            pull_all<L, S>(fin, g, x, y, z, cell, ph, df);
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i) df[i] = pull_one<L, S>(fin, g, x, y, z, cell, i, ph.sc);
        }
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) df[i] = (T)0;
    }

    // ---- 2. moments (Eq. 5): rho = 1 + sum d_i, rho u = j + F/2
    T drho = 0, jx = 0, jy = 0, jz = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        drho += df[i];
        if (L::ex(i)) jx += L::ex(i) * df[i];
        if (L::ey(i)) jy += L::ey(i) * df[i];
        if (L::ez(i)) jz += L::ez(i) * df[i];
    }
    const T rho = (T)1 + drho;
    const T irho = (T)1 / rho;
    const T ux = (jx + (T)0.5 * ph.F[0]) * irho;
    const T uy = (jy + (T)0.5 * ph.F[1]) * irho;
    const T uz = (jz + (T)0.5 * ph.F[2]) * irho;
    if (active && !(rho > (T)0)) atomicOr(flags, 1);

#pragma unroll
    for (int j = 0; j < kRecWords; ++j) {
        const int w = tid + j * kThreads;
        if (w < nwords) srec[w] = rw[j];
    }

    // ---- 3. candidates reaching this row: solid fractions and u_s moments of the cell
    const T cx = (T)((int)threadIdx.x - L::REC_X), cy = (T)threadIdx.y, cz = (T)threadIdx.z;
    const T xmax = (T)(min(L::TX, g.n[0] - x0) - 1);
    T seps = 0, mx = 0, my = 0, mz = 0, Mxx = 0, Myy = 0, Mzz = 0, Mxy = 0, Mxz = 0, Myz = 0;
    unsigned long long wmask = 0ull;     // relevant candidates of this row (normal tiles)
    T eslot[NSLOT] = {};                 // eps of the first relevant candidates, for step 6
    int nk = cnt;
    for (int ch = 0; ch < nchunk; ++ch) {
        if (ovf) {
            nk = min(cap, pd.n - ch * cap);
            __syncthreads();
            if (tid < nk) write_record<L, T>(srec + tid * RW, g, pd, ch * cap + tid, x0, y0, z0);
        }
        __syncthreads();
        int js = 0;
        for (int kb = 0; kb < nk; kb += 32) {
            const int k = kb + lane;
            bool rel = false;
            if (k < nk) {
                const Vec4<T> a = ld4<T>(srec + k * RW);
                rel = row_hits<L, T>(g, a.x + (T)L::REC_X, a.y, a.z, a.w + ph.h, cy, cz, xmax);
            }
            unsigned bal = __ballot_sync(kFull, rel);
            if (!ovf) wmask |= (unsigned long long)bal << kb;
            while (bal) {
                const int kk = kb + __ffs(bal) - 1;
                bal &= bal - 1u;
                const T *rk = srec + kk * RW;
                const Vec4<T> a = ld4<T>(rk);
                const Vec4<T> b = ld4<T>(rk + 4);      // f(r), Ux, Uy, Uz
                T dx, dy, dz;
                cand_arm<L, T>(g, cx, cy, cz, a.x, a.y, a.z, dx, dy, dz);
                const T e = active ? shell_eps<T>(dx * dx + dy * dy + dz * dz, a.w, b.x, ph.h) : (T)0;
                if (!ovf) {
#pragma unroll
                    for (int q = 0; q < NSLOT; ++q) if (js == q) eslot[q] = e;
                }
                ++js;
                if (e > (T)0) {
                    const Vec4<T> c = ld4<T>(rk + 8);  // Ox, Oy, Oz, id
                    // u_s = U + Omega x (x_n - X_p)
                    const T usx = b.y + c.y * dz - c.z * dy;
                    const T usy = b.z + c.z * dx - c.x * dz;
                    const T usz = (L::D == 3) ? b.w + c.x * dy - c.y * dx : (T)0;
                    // modified scheme weights by eps_s (normalised below); original by B(eps_s)
                    const T wgt = (PSC == 0) ? e : e * ph.tmh / (((T)1 - e) + ph.tmh);
                    seps += wgt;
                    mx += wgt * usx; my += wgt * usy; mz += wgt * usz;
                    Mxx += wgt * usx * usx; Myy += wgt * usy * usy; Mxy += wgt * usx * usy;
                    if (L::D == 3) { Mzz += wgt * usz * usz; Mxz += wgt * usx * usz; Myz += wgt * usy * usz; }
                }
            }
        }
    }

    // ---- 4. weights: eps_n = min(1, sum eps) (Table 1 Step 5), B_n by Eq. 9 at eps_n,
    //         B_{n,s} = B_n eps_s / sum eps = cB eps_s (Eq. 13; cells with overlapping
    //         fractions keep B_n = 1). Original scheme: B_n = sum_s B(eps_s) (Eq. 8).
    const bool any_solid = __any_sync(kFull, seps > (T)0);
    T Bn = 0, cB = 0;
    if (any_solid && seps > (T)0) {
        if (PSC == 0) {
            if (seps < (T)1) {
                const T c = ph.tmh / (((T)1 - seps) + ph.tmh);
                Bn = seps * c;
                cB = c;
            } else {
                Bn = (T)1;
                cB = (T)1 / seps;
            }
        } else {
            Bn = seps;
            cB = (T)1;
        }
        mx *= cB; my *= cB; mz *= cB;
        Mxx *= cB; Myy *= cB; Mzz *= cB; Mxy *= cB; Mxz *= cB; Myz *= cB;
    }

    // ---- 5. collision (Eq. 2-4, 10, 12) in deviation form, then store
    const T uu = ux * ux + uy * uy + uz * uz;
    const T uF = ux * ph.F[0] + uy * ph.F[1] + uz * ph.F[2];
    if (!any_solid) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const T w = (T)weight<L>(i);
            const T eu = L::ex(i) * ux + L::ey(i) * uy + L::ez(i) * uz;
            const T eF = L::ex(i) * ph.F[0] + L::ey(i) * ph.F[1] + L::ez(i) * ph.F[2];
            const T dfeq = w * (drho + rho * ((T)3 * eu + (T)4.5 * eu * eu - (T)1.5 * uu));
            const T fi = ph.guo * w * ((T)3 * (eF - uF) + (T)9 * eu * eF);
            const T out = df[i] - ph.omega * (df[i] - dfeq) + fi;
            if (active) Store<S>::st(fout, PSC_IDX((long long)i * N + cell, Q * N, CHK_POP), out, ph.sc);
        }
    } else {
        const T trM = Mxx + Myy + Mzz;
        const T omB = (T)1 - Bn;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int o = opp<L>(i);
            const T w = (T)weight<L>(i);
            const T ex = (T)L::ex(i), ey = (T)L::ey(i), ez = (T)L::ez(i);
            const T eu = ex * ux + ey * uy + ez * uz;
            const T eF = ex * ph.F[0] + ey * ph.F[1] + ez * ph.F[2];
            const T sym = drho + rho * ((T)4.5 * eu * eu - (T)1.5 * uu);
            const T dfeq = w * (sym + rho * (T)3 * eu);
            const T dfeq_o = w * (sym - rho * (T)3 * eu);
            const T fi = ph.guo * w * ((T)3 * (eF - uF) + (T)9 * eu * eF);
            const T em = ex * mx + ey * my + ez * mz;
            const T eMe = ex * ex * Mxx + ey * ey * Myy + ez * ez * Mzz +
                          (T)2 * (ex * ey * Mxy + ex * ez * Mxz + ey * ez * Myz);
            const T sfe = w * (Bn * drho + rho * ((T)3 * em + (T)4.5 * eMe - (T)1.5 * trM));
            const T out = df[i] - omB * ph.omega * (df[i] - dfeq) + Bn * (df[o] - dfeq_o - df[i]) +
                          sfe + omB * fi;
            if (active) Store<S>::st(fout, PSC_IDX((long long)i * N + cell, Q * N, CHK_POP), out, ph.sc);
        }
    }

    // ---- 6. force and torque (Eq. 14; Eq. 11 in original mode):
    //         F_p -= B_{n,s} (rho u_s + F/2 - j),  T_p -= (x_n - X_p) x (same)
    const bool solid = active && seps > (T)0;
    const T px = (T)0.5 * ph.F[0] - jx, py = (T)0.5 * ph.F[1] - jy, pz = (T)0.5 * ph.F[2] - jz;
    if (!ovf && lane == 0) s_mask[warp] = any_solid ? wmask : 0ull;
    if (any_solid) {
        for (int ch = 0; ch < nchunk; ++ch) {
            if (ovf) {
                nk = min(cap, pd.n - ch * cap);
                __syncwarp();
                // overflow tiles: each warp restages nothing; records come from global memory
            }
            int js = 0;
            for (int kb = 0; kb < nk; kb += 32) {
                const int k = kb + lane;
                bool rel;
                T ovr[RW];
                if (!ovf) {
                    rel = (wmask >> k) & 1ull;
                } else {
                    rel = false;
                    if (k < nk) {
                        write_record<L, T>(ovr, g, pd, ch * cap + k, x0, y0, z0);
                        rel = row_hits<L, T>(g, ovr[R_PX] + (T)L::REC_X, ovr[R_PY], ovr[R_PZ], ovr[R_R] + ph.h, cy, cz, xmax);
                    }
                }
                unsigned bal = __ballot_sync(kFull, rel);
                while (bal) {
                    const int src = __ffs(bal) - 1;
                    const int kk = kb + src;
                    bal &= bal - 1u;
                    T a[RW];
                    if (!ovf) {
#pragma unroll
                        for (int q = 0; q < RW; ++q) a[q] = srec[kk * RW + q];
                    } else {
#pragma unroll
                        for (int q = 0; q < RW; ++q) a[q] = __shfl_sync(kFull, ovr[q], src);
                    }
                    T v[NC];
#pragma unroll
                    for (int q = 0; q < NC; ++q) v[q] = (T)0;
                    if (solid) {
                        T dx, dy, dz;
                        cand_arm<L, T>(g, cx, cy, cz, a[R_PX], a[R_PY], a[R_PZ], dx, dy, dz);
                        T e = (T)0;
                        if (!ovf && js < NSLOT) {
#pragma unroll
                            for (int q = 0; q < NSLOT; ++q) if (js == q) e = eslot[q];
                        } else {
                            e = shell_eps<T>(dx * dx + dy * dy + dz * dz, a[R_R], a[R_FR], ph.h);
                        }
                        if (e > (T)0) {
                            const T usx = a[R_UX] + a[R_OY] * dz - a[R_OZ] * dy;
                            const T usy = a[R_UY] + a[R_OZ] * dx - a[R_OX] * dz;
                            const T usz = (L::D == 3) ? a[R_UZ] + a[R_OX] * dy - a[R_OY] * dx : (T)0;
                            const T Bs = (PSC == 0) ? cB * e : Bn;
                            const T dPx = Bs * (rho * usx + px);
                            const T dPy = Bs * (rho * usy + py);
                            const T dPz = (L::D == 3) ? Bs * (rho * usz + pz) : (T)0;
                            if (L::D == 2) {
                                v[0] = dPx; v[1] = dPy; v[2] = dx * dPy - dy * dPx;
                            } else {
                                v[0] = dPx; v[1] = dPy; v[2] = dPz;
                                v[3] = dy * dPz - dz * dPy;
                                v[4] = dz * dPx - dx * dPz;
                                v[5] = dx * dPy - dy * dPx;
                            }
                        }
                    }
                    ++js;
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
                        for (int q = 0; q < NC; ++q) v[q] += __shfl_xor_sync(kFull, v[q], off);
                    }
                    if (lane == 0) {
                        if (!ovf) {
#pragma unroll
                            for (int q = 0; q < NC; ++q) part[((size_t)warp * cap + kk) * NC + q] = v[q];
                        } else {
                            const int pid = (int)PSC_IDX(bits_id(a[R_ID]), pd.n, CHK_PART);
#pragma unroll
                            for (int q = 0; q < NC; ++q) {
                                if (v[q] == (T)0) continue;
                                double *dst;
                                if (L::D == 2) dst = (q < 2) ? &pd.F[3 * pid + q] : &pd.T[3 * pid + 2];
                                else dst = (q < 3) ? &pd.F[3 * pid + q] : &pd.T[3 * pid + q - 3];
                                atomicAdd(dst, -(double)v[q]);
                            }
                        }
                    }
                }
            }
        }
    }
    if (ovf) return;   // uniform over the block
    __syncthreads();
    // tile totals in a fixed warp order, one FP64 atomic per particle component
    for (int idx = tid; idx < cnt * NC; idx += kThreads) {
        const int k = idx / NC, q = idx - k * NC;
        T sum = 0;
        bool any = false;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            if ((s_mask[w] >> k) & 1ull) { sum += part[((size_t)w * cap + k) * NC + q]; any = true; }
        }
        if (any && sum != (T)0) {
            const int p = bits_id(srec[k * RW + R_ID]);
            double *dst;
            if (L::D == 2) dst = (q < 2) ? &pd.F[3 * p + q] : &pd.T[3 * p + 2];
            else dst = (q < 3) ? &pd.F[3 * p + q] : &pd.T[3 * p + q - 3];
            atomicAdd(dst, -(double)sum);
        }
    }
}

#include "psc_pair.cuh"
#include "psc_pair16.cuh"

// Tiles with more candidates than the block holds (rare): the exact chunked path over all
// particles, one block per tile of the overflow list. Its tiles are no other kernel's, so after
// k_step (which starts it early, see launch_step_t; by then the lists are there) it works beside it
// and only ends after it. With no such tile its launch then costs what its end does.
template <class L, typename S, int PSC>
__global__ void __launch_bounds__(kThreads, 1)
k_collide_overflow(const S *__restrict__ fin, S *__restrict__ fout, Geom g, PhysT<typename Store<S>::T> ph,
                   Tiles tl, Parts pd, int *flags) {
    using T = typename Store<S>::T;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long s_mask[kWarps];
    const long long ntiles = (long long)g.nt[0] * g.nt[1] * g.nt[2];
    const int novf = tl.stats[2];
    pdl_launch();
    for (int it = blockIdx.x; it < novf; it += gridDim.x) {
        psc_tile<L, S, PSC>(tl.order[2 * ntiles + it], fin, fout, g, ph, tl, pd, flags, reinterpret_cast<T *>(smem), s_mask);
        __syncthreads();
    }
    pdl_wait();
    // the pair kernel before this one has finished: clear its work counters
    if ((sizeof(S) == 2 || tl.keep) && blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0 && threadIdx.z == 0) {
        tl.stats[3] = 0;
        tl.stats[6] = 0;
    }
}

// Contexts with an open, inlet or outlet face, by the single-cell path whose pull classifies each
// face: SOLID the list of tiles with candidates (blocks striding over it), else those without
// (every tile when there are no particles; a block each). Apart, the tiles without need a third of
// the registers, so three blocks instead of one share an SM. Few tiles with candidates leave most
// of the chip idle, so the other launch starts as soon as this one's blocks have (its tiles are
// others) and ends after it; a block per tile evens out the SMs where those still run. A step of
// 120 x 60 x 60 FP32 with one sphere: one kernel for both 104 us, one after the other 66, now 51
// (58 with striding blocks); 500 x 300 FP64 with one disc 90, 105 and 88 (94).
template <class L, typename S, int PSC, bool SOLID>
__global__ void __launch_bounds__(kThreads, SOLID ? 1 : (sizeof(S) == 8 ? 2 : 3))
k_collide_faces(const S *__restrict__ fin, S *__restrict__ fout, Geom g, PhysT<typename Store<S>::T> ph,
                Tiles tl, Parts pd, int *flags) {
    using T = typename Store<S>::T;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long s_mask[kWarps];
    const unsigned ntiles = (unsigned)g.nt[0] * (unsigned)g.nt[1] * (unsigned)g.nt[2];
    if (SOLID) pdl_launch();      // what both read was there before this launch, and their tiles differ
    const unsigned n = SOLID ? (unsigned)tl.stats[4] : (pd.n > 0 ? (unsigned)tl.stats[5] : ntiles);
    for (unsigned it = blockIdx.x; it < n; it += gridDim.x) {
        const unsigned tile = SOLID ? tl.order[it] : (pd.n > 0 ? tl.order[ntiles + it] : it);
        psc_tile<L, S, PSC, true, !SOLID>(tile, fin, fout, g, ph, tl, pd, flags, reinterpret_cast<T *>(smem), s_mask);
        __syncthreads();
    }
    if (!SOLID) pdl_wait();       // not done before the other is
}

// ---------------------------------------------------------------- gather / set kernels
template <class L, typename S>
__global__ void k_gather(const S *__restrict__ fin, Geom g, PhysT<typename Store<S>::T> ph, double *f_out) {
    const long long cell = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (cell >= g.ncell) return;
    const int x = (int)(cell % g.n[0]);
    const int y = (int)((cell / g.n[0]) % g.n[1]);
    const int z = (int)(cell / ((long long)g.n[0] * g.n[1]));
    typename Store<S>::T df[L::Q];
    pull_all<L, S>(fin, g, x, y, z, cell, ph, df);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) f_out[(long long)i * g.ncell + cell] = weight<L>(i) + (double)df[i];
}

// A float as a double by integer operations (the FP64 pipe converts at 1/64 of the FP32
// rate); values below the normal range become 0.
__device__ __forceinline__ double widen(const float v) {
    const unsigned b = __float_as_uint(v), a = b & 0x7fffffffu;
    const unsigned hi = (b & 0x80000000u) | ((a >> 3) + 0x38000000u);
    return a < 0x00800000u ? 0.0 : __hiloint2double((int)hi, (int)(a << 29));
}

// The four moments of Eq. 5 (drho, j) of a cell in FP64, added one after the other.
template <class L, typename T>
__device__ __forceinline__ void moments_f64(const T *df, double &drho, double *j) {
    drho = j[0] = j[1] = j[2] = 0.0;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const double d = (double)df[i];
        drho += d;
        if (L::ex(i)) j[0] += L::ex(i) > 0 ? d : -d;
        if (L::ey(i)) j[1] += L::ey(i) > 0 ? d : -d;
        if (L::ez(i)) j[2] += L::ez(i) > 0 ? d : -d;
    }
}
template <class L, typename T>
__device__ __noinline__ void moments_f64_cold(const T *df, double &drho, double *j) { moments_f64<L, T>(df, drho, j); }

// The same sums from FP32 values, no less accurate than in FP64 but almost all on the FP32
// pipe (error-free vector transformation of Rump, Ogita and Oishi, "Accurate floating-point
// summation", 2008): with max |d| < 2^k every d is cut into q1 + q2 + r, q1 a multiple of
// 2^(k-17), q2 of 2^(k-34), |r| <= 2^(k-34), by adding and subtracting 2^(k+7) and 2^(k-10).
// The at most 19 q1 of a sum (and likewise the q2) have an exact FP32 sum, whatever the signs;
// the r's sum, below 2^(k-29), is rounded in FP32 by at most 2^(k-54) an addition. Two FP64
// additions put a moment together. rhof is the density with three roundings in FP32 (all three
// parts count where it is far below 1: without the q2, a density of 0.02 was off by 1e-4 of itself
// and the velocity by 2e-13). Returns false, with nothing written, for values outside [2^-60, 2^10] (or not finite).
template <class L>
__device__ __forceinline__ bool moments_split(const float *df, double &drho, double *j, float &rhof) {
    float m = 0.0f;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) m = fmaxf(m, fabsf(df[i]));
    if (!(m <= 0x1p10f) || (m < 0x1p-60f && m > 0.0f)) return false;
    const unsigned eb = __float_as_uint(m) & 0x7f800000u;      // 2^(k-1) <= m < 2^k
    const float s1 = m > 0.0f ? __uint_as_float(eb + (8u << 23)) : 1.0f;
    const float s2 = __fmul_rn(s1, 0x1p-17f);
    float t[3][4] = {};
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const float q1 = __fsub_rn(__fadd_rn(df[i], s1), s1), r1 = __fsub_rn(df[i], q1);
        const float q2 = __fsub_rn(__fadd_rn(r1, s2), s2);
        const float q[3] = {q1, q2, __fsub_rn(r1, q2)};
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            t[l][0] = __fadd_rn(t[l][0], q[l]);
            if (L::ex(i)) t[l][1] = __fadd_rn(t[l][1], L::ex(i) > 0 ? q[l] : -q[l]);
            if (L::ey(i)) t[l][2] = __fadd_rn(t[l][2], L::ey(i) > 0 ? q[l] : -q[l]);
            if (L::ez(i)) t[l][3] = __fadd_rn(t[l][3], L::ez(i) > 0 ? q[l] : -q[l]);
        }
    }
    if (!(t[0][0] == t[0][0])) return false;                   // fmaxf drops NaN; every d is in t[][0]
    double o[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) o[c] = (c <= L::D) ? (widen(t[0][c]) + widen(t[1][c])) + widen(t[2][c]) : 0.0;
    drho = o[0]; j[0] = o[1]; j[1] = o[2]; j[2] = o[3];
    rhof = 1.0f + __fadd_rn(__fadd_rn(t[0][0], t[1][0]), t[2][0]);
    return true;
}

// Density and force-shifted velocity (Eq. 5) of every cell in FP64, one block per lattice
// tile, one warp per row. Bound by the FP64 pipe (1/64 of the FP32 rate): the moments of FP32
// values are summed by moments_split, and u = (j + F/2) / rho shares one reciprocal (one
// Newton step on the FP32 one, off by at most 2^-18 for densities above 2^-6, then per component the
// quotient and one residual correction, which leaves it correctly rounded but for rare ties): 23 FP64 operations a cell where 19
// conversions, 95 additions and three divisions stood before. The three components leave
// through shared memory, a row's 96 doubles in order. 256^3 D3Q19: 4.03 -> 0.82 ms in FP32,
// 5.65 -> 0.82 ms in FP16 (its bytes take 0.27 and 0.17 ms); 2048^2 D2Q9 FP32: 0.66 -> 0.20 ms.
template <class L, typename S, bool FACES>
__global__ void __launch_bounds__(kThreads)
k_macro(const S *__restrict__ fin, Geom g, PhysT<typename Store<S>::T> ph, double F0, double F1, double F2,
        double *rho_out, double *u_out) {
    using T = typename Store<S>::T;
    __shared__ double s_u[kWarps][3 * 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // grid (nt0 * nt1, 1, nt2); a warp takes 32 cells of a row
    const int ty = (int)(blockIdx.x / (unsigned)g.nt[0]), row_of = warp / (L::TX / 32);
    const int x0 = (int)(blockIdx.x - (unsigned)ty * (unsigned)g.nt[0]) * L::TX + 32 * (warp % (L::TX / 32));
    const int x = x0 + lane, y = ty * L::TY + row_of % L::TY, z = (int)blockIdx.z * L::TZ + row_of / L::TY;
    if (x0 >= g.n[0] || y >= g.n[1] || z >= g.n[2]) return;       // the whole warp
    const bool in = x < g.n[0];
    const long long row = (long long)g.n[0] * (y + (long long)g.n[1] * z);
    const long long cell = row + x;
    T df[L::Q];
    if (FACES) {
        if (in) pull_all<L, S>(fin, g, x, y, z, cell, ph, df);
    } else {
        const bool interior = x0 >= 1 && x0 + 32 < g.n[0] && y >= 1 && y + 1 < g.n[1] &&
                              (L::D == 2 || (z >= 1 && z + 1 < g.n[2]));
        pull_q<L, S>(fin, g, x, y, z, cell, interior, in, ph.sc, df);
    }
    const int count = min(32, g.n[0] - x0);
    if (in) {
        double drho, j[3];
        float rhof = 0.0f;
        bool split = false;
        if constexpr (sizeof(T) == 4) {
            split = moments_split<L>(df, drho, j, rhof);
            if (!split) moments_f64_cold<L, T>(df, drho, j);
        } else {
            moments_f64<L, T>(df, drho, j);
        }
        const double rho = 1.0 + drho;
        if (rho_out) rho_out[cell] = rho;
        if (u_out) {
            const double F[3] = {F0, F1, F2};
            if (split && rhof > 0x1p-6f && rhof < 0x1p6f) {
                const double r0 = widen(1.0f / rhof);
                const double r = fma(fma(-rho, r0, 1.0), r0, r0);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    double v = 0.0;
                    if (a < L::D || F[a] != 0.0) {
                        const double n = F[a] != 0.0 ? j[a] + 0.5 * F[a] : j[a];
                        const double q = n * r;
                        v = fma(fma(-q, rho, n), r, q);
                    }
                    s_u[warp][3 * lane + a] = v;
                }
            } else {
#pragma unroll
                for (int a = 0; a < 3; ++a) s_u[warp][3 * lane + a] = (j[a] + 0.5 * F[a]) / rho;
            }
        }
    }
    if (!u_out) return;
    __syncwarp();
    double *dst = u_out + 3 * (row + x0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int w = lane + 32 * k;
        if (w < 3 * count) dst[w] = s_u[warp][w];
    }
}

// Inverse of the pull: the stored post-collision value f^+_i(x) is the pre-collision
// f_i(x + e_i), or f_{-i}(x) when x + e_i lies beyond a wall.
template <class L, typename S>
__global__ void k_set(const double *__restrict__ f, S *__restrict__ fout, Geom g,
                      PhysT<typename Store<S>::T> ph) {
    const long long cell = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (cell >= g.ncell) return;
    const int xc[3] = {(int)(cell % g.n[0]), (int)((cell / g.n[0]) % g.n[1]),
                       (int)(cell / ((long long)g.n[0] * g.n[1]))};
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const int e[3] = {L::ex(i), L::ey(i), L::ez(i)};
        int d[3];
        bool wall = false, leaves = false;
        for (int a = 0; a < 3; ++a) {
            d[a] = xc[a] + e[a];
            if (d[a] < 0 || d[a] >= g.n[a]) {
                const int kind = face_kind(g, a, d[a] < 0 ? 0 : 1);
                if (kind == FACE_PERIODIC) d[a] += (d[a] < 0) ? g.n[a] : -g.n[a];
                else if (kind == FACE_WALL) wall = true;
                else leaves = true;
            }
        }
        double v;
        if (wall) v = f[(long long)opp<L>(i) * g.ncell + cell];
        else if (leaves) v = f[(long long)i * g.ncell + cell];     // leaves the lattice: never pulled
        else v = f[(long long)i * g.ncell + d[0] + (long long)g.n[0] * (d[1] + (long long)g.n[1] * d[2])];
        Store<S>::st(fout, PSC_IDX((long long)i * g.ncell + cell, L::Q * g.ncell, CHK_POP), (typename Store<S>::T)(v - weight<L>(i)), ph.sc);
    }
}

// Blocks of a persistent grid: as many as stay resident on all SMs (never more than the
// work items). The occupancy query is cached per kernel and shared-memory size.
template <typename K>
inline cudaError_t persistent_blocks(K kern, size_t smem, long long work, unsigned &blocks, int threads = kThreads,
                                     int *per_sm = nullptr) {
    static thread_local const void *c_kern = nullptr;
    static thread_local size_t c_smem = (size_t)-1;
    static thread_local int c_per = 0, c_threads = 0;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (c_smem != smem || c_kern != (const void *)kern || c_threads != threads) {
        int per = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem);
        if (e != cudaSuccess) return e;
        c_per = per > 0 ? per : 1;
        c_smem = smem;
        c_kern = (const void *)kern;
        c_threads = threads;
    }
    const long long b = (long long)sms * c_per;
    blocks = (unsigned)(b < work ? b : (work > 0 ? work : 1));
    if (per_sm) *per_sm = c_per;
    return cudaSuccess;
}

// The overflow-tile kernel (tiles with more candidates than the step's kernel keeps), which
// also clears that kernel's work counters for the next launch.
template <class L, typename S, int PSC>
cudaError_t launch_overflow(const void *fin, void *fout, const Geom &g, const PhysT<typename Store<S>::T> &pt,
                            const Tiles &tl, const Parts &pd, int *flags, cudaStream_t s) {
    using T = typename Store<S>::T;
    constexpr int NC = (L::D == 2) ? 3 : 6;
    const size_t osmem = cs_smem_bytes<T>(tl.cap, NC);
    auto okern = k_collide_overflow<L, S, PSC>;
    if (osmem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(okern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)osmem);
        if (e != cudaSuccess) return e;
    }
    const dim3 block(L::TX, L::TY, L::TZ);
    if (sizeof(S) != 2 && !tl.keep) return launch_pdl(okern, dim3(32), block, osmem, s, (const S *)fin, (S *)fout, g, pt, tl, pd, flags);
    okern<<<32, block, osmem, s>>>((const S *)fin, (S *)fout, g, pt, tl, pd, flags);
    return cudaGetLastError();
}

// Fluid-tile blocks per SM when they follow the particle tiles beside the caller's next
// kernels (a deferred join). 20 coupled steps of 2048^2 with 5000 discs, 5 of 4096^2 with 20000,
// ms: 2 blocks 2.98 and 2.84, 3 2.93 and 2.63, 4 2.98 and 2.58, 5 3.17 and 2.73 (the
// caller's kernels find no room beside them).
constexpr int kDeferF = 3;

// One launch of the step's kernel over the lists `which` (blocks_per_sm > 0 limits it).
template <class L, typename S, int PSC, bool SOLID, bool VEC>
cudaError_t launch_step_t(const void *fin, void *fout, const Geom &g, const PhysT<typename Store<S>::T> &pt,
                          const Tiles &tl, const Parts &pd, int *flags, int which, int blocks_per_sm, cudaStream_t s) {
    auto kern = k_step<L, S, PSC, SOLID, VEC>;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const long long ntiles = (long long)g.nt[0] * g.nt[1] * g.nt[2];
    // a whole tile per item where every warp of a full chip gets many (256^3 with 2000 spheres, FP32:
    // 421 us against 456), else a unit (128^3 with 200 62 against 64, 1024^2 FP64 327 against 368,
    // 777 x 453 15.6 against 24; 2048^2 FP32 65.7 and 65.0); few items go to blocks of one warp,
    // spread over the SMs
    const int shift = ntiles >= 16LL * 16 * sms ? 0 : 2;
    const long long items = ntiles << shift;
    const int threads = items <= 8LL * sms ? 32 : kPThreads;
    unsigned nb = 0;
    e = persistent_blocks(kern, 0, (items + threads / 32 - 1) / (threads / 32), nb, threads);
    if (e != cudaSuccess) return e;
    if (blocks_per_sm > 0 && nb > (unsigned)(blocks_per_sm * sms)) nb = (unsigned)(blocks_per_sm * sms);
    const Dirs<L, S> f(fin, fout, g);
    if (which != kFluidTiles)
        return launch_pdl(kern, dim3(nb), dim3((unsigned)threads), 0, s, f, g, pt, tl, pd, flags, tl.work, which, shift);
    // on the second stream after an event: the usual order, and counters of its own
    kern<<<nb, threads, 0, s>>>(f, g, pt, tl, pd, flags, tl.work + kCounters * kCounterStride, which, shift);
    return cudaGetLastError();
}

// The step of a lattice without particles; few units go to blocks of one warp, spread over the SMs.
template <class L, typename S, bool VEC>
cudaError_t launch_fluid_t(const void *fin, void *fout, const Geom &g, const PhysT<typename Store<S>::T> &pt, int *flags,
                           cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    static_assert(kUnits % kPWarps == 0, "a block's units end with the lattice's");
    const long long units = (long long)g.nt[0] * g.nt[1] * g.nt[2] * kUnits;
    const int threads = units <= 8LL * sms ? 32 : kPThreads;
    return launch_pdl(k_fluid<L, S, VEC>, dim3((unsigned)(units / (threads / 32))), dim3((unsigned)threads), 0, s,
                      Dirs<L, S>(fin, fout, g), g, pt, flags);
}

// One collide-stream step. Without particles: the fluid kernel over every tile. With
// particles: one kernel over the tiles with candidates and then those without, and the
// overflow kernel. In a coupled step (ov->defer; 2D FP32) the tiles with
// candidates and the overflow tiles first, then those without on the second stream, a few
// blocks per SM, beside the caller's next kernels.
template <class L, typename S, int PSC, bool VEC>
cudaError_t launch_collide_stream_t(const void *fin, void *fout, const Geom &g, const Phys &ph,
                                    const Tiles &tl, const Parts &pd, int *flags, cudaStream_t s,
                                    Overlap *ov) {
    using T = typename Store<S>::T;
    const PhysT<T> pt = make_phys<T>(ph, L::Q);
    if (pd.n == 0) return launch_fluid_t<L, S, VEC>(fin, fout, g, pt, flags, s);
    const bool defer = ov && ov->aux && ov->defer && L::D == 2 && sizeof(T) == 4;
    cudaError_t e = launch_step_t<L, S, PSC, true, VEC>(fin, fout, g, pt, tl, pd, flags,
                                                              defer ? kParticleTiles : kBothLists, 0, s);
    if (e == cudaSuccess && may_overflow(tl.cap, pd.n)) e = launch_overflow<L, S, PSC>(fin, fout, g, pt, tl, pd, flags, s);
    if (e != cudaSuccess || !defer) return e;
    e = cudaEventRecord(ov->fork, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(ov->aux, ov->fork, 0);
    if (e == cudaSuccess)
        e = launch_step_t<L, S, 0, false, VEC>(fin, fout, g, pt, tl, pd, flags, kFluidTiles, kDeferF, ov->aux);
    if (e == cudaSuccess) e = cudaEventRecord(ov->join, ov->aux);
    if (e == cudaSuccess) ov->deferred = 1;
    return e;
}

// Registers a block of `threads` holds (allocated per warp in units of 8 per thread).
template <typename K>
inline cudaError_t block_registers(K kern, int threads, int &regs) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    regs = (e == cudaSuccess) ? ((fa.numRegs + 7) / 8 * 8) * threads : 0;
    return e;
}

// 16-bit storage (and the adjoint's steps in FP32). Without particles: the fluid kernel over every
// tile. With particles in 2D: the particle-tile kernel (4 blocks per SM) and the fluid-tile
// kernel (3 blocks per SM) side by side on two streams, which together fill
// each SM's register file, so the issue-bound particle tiles and the DRAM-bound fluid tiles
// share every SM for the whole step; without a second stream, one after the other. In 3D
// the particle-tile kernel holds all the registers an SM has, and takes the
// fluid tiles itself once its own are done. Then the overflow kernel.
template <class L, typename S, int PSC>
cudaError_t launch_collide_stream16(const void *fin, void *fout, const Geom &g, const Phys &ph,
                                    const Tiles &tl, const Parts &pd, int *flags, cudaStream_t s,
                                    Overlap *ov) {
    using T = typename Store<S>::T;
    constexpr bool kSteal = L::D == 3;
    // blocks per SM side by side (2D): 4 x 128 threads x 80 registers + 3 x 128 x 64 = 64 K
    constexpr int kSideP = 4, kSideF = 3, kDeferF16 = 2;
    const size_t smem = h16::pair_smem_bytes<L, T>();
    auto kern = h16::k_collide_stream<L, S, PSC, kSteal>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const long long ntiles = (long long)g.nt[0] * g.nt[1] * g.nt[2];
    const PhysT<T> pt = make_phys<T>(ph, L::Q);
    const Dirs<L, S> f(fin, fout, g);
    const bool hasF = ph.body_force[0] != 0.0 || ph.body_force[1] != 0.0 || ph.body_force[2] != 0.0;
    auto fkern = hasF ? h16::k_fluid_pair<L, S, true> : h16::k_fluid_pair<L, S, false>;
    const dim3 pblock(32, kPWarps);
    if (pd.n == 0) {
        fkern<<<dim3(g.nt[0], g.nt[1], g.nt[2]), pblock, 0, s>>>(f, g, pt, tl, 0, flags);
        return cudaGetLastError();
    }
    cudaError_t e;
    unsigned nb = 0;
    bool side = false;
    int nsm = 0;
    if (!kSteal && ov && ov->aux) {
        int dev = 0, rf_sm = 0, rp = 0, rf = 0, per = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&rf_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
        if (e == cudaSuccess) e = block_registers(kern, kPThreads, rp);
        if (e == cudaSuccess) e = block_registers(fkern, kPThreads, rf);
        if (e == cudaSuccess) e = persistent_blocks(kern, smem, ntiles, nb, kPThreads, &per);
        if (e != cudaSuccess) return e;
        side = per >= kSideP && kSideP * rp + kSideF * rf <= rf_sm;
    }
    if (side && ov->defer) {
        e = persistent_blocks(kern, smem, ntiles, nb, kPThreads);
        if (e != cudaSuccess) return e;
        kern<<<nb, pblock, smem, s>>>(f, g, pt, tl, pd, flags);
        e = launch_overflow<L, S, PSC>(fin, fout, g, pt, tl, pd, flags, s);
        if (e == cudaSuccess) e = cudaEventRecord(ov->fork, s);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(ov->aux, ov->fork, 0);
        if (e != cudaSuccess) return e;
        fkern<<<nsm * kDeferF16, pblock, 0, ov->aux>>>(f, g, pt, tl, pd.n, flags);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaEventRecord(ov->join, ov->aux);
        if (e == cudaSuccess) ov->deferred = 1;
        return e;
    }
    if (side) {
        e = cudaEventRecord(ov->fork, s);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(ov->aux, ov->fork, 0);
        if (e != cudaSuccess) return e;
        kern<<<nsm * kSideP, pblock, smem, s>>>(f, g, pt, tl, pd, flags);
        fkern<<<nsm * kSideF, pblock, 0, ov->aux>>>(f, g, pt, tl, pd.n, flags);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaEventRecord(ov->join, ov->aux);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ov->join, 0);
        if (e != cudaSuccess) return e;
    } else {
        if (!kSteal) {
            e = persistent_blocks(fkern, 0, ntiles, nb, kPThreads);
            if (e != cudaSuccess) return e;
            fkern<<<nb, pblock, 0, s>>>(f, g, pt, tl, pd.n, flags);
        }
        e = persistent_blocks(kern, smem, ntiles, nb, kPThreads);
        if (e != cudaSuccess) return e;
        kern<<<nb, pblock, smem, s>>>(f, g, pt, tl, pd, flags);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return launch_overflow<L, S, PSC>(fin, fout, g, pt, tl, pd, flags, s);
}

template <class L, typename S, int PSC>
cudaError_t launch_faces_t(const void *fin, void *fout, const Geom &g, const Phys &ph, const Tiles &tl, const Parts &pd,
                           int *flags, cudaStream_t s) {
    using T = typename Store<S>::T;
    const PhysT<T> pt = make_phys<T>(ph, L::Q);
    const dim3 block(L::TX, L::TY, L::TZ);
    const long long ntiles = (long long)g.nt[0] * g.nt[1] * g.nt[2];
    unsigned nb = 0;
    if (pd.n > 0) {
        auto kern = k_collide_faces<L, S, PSC, true>;
        const size_t smem = cs_smem_bytes<T>(tl.cap, L::D == 2 ? 3 : 6);
        cudaError_t e = cudaSuccess;
        if (smem > 48 * 1024) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) e = persistent_blocks(kern, smem, ntiles, nb, kThreads);
        if (e != cudaSuccess) return e;
        kern<<<nb, block, smem, s>>>((const S *)fin, (S *)fout, g, pt, tl, pd, flags);
    }
    auto kern = k_collide_faces<L, S, PSC, false>;
    if (pd.n > 0) return launch_pdl(kern, dim3((unsigned)ntiles), block, 0, s, (const S *)fin, (S *)fout, g, pt, tl, pd, flags);
    kern<<<(unsigned)ntiles, block, 0, s>>>((const S *)fin, (S *)fout, g, pt, tl, pd, flags);
    return cudaGetLastError();
}

template <class L, typename S, int PSC>
cudaError_t launch_collide_stream_l(const void *fin, void *fout, const Geom &g, const Phys &ph, const Tiles &tl,
                                    const Parts &pd, int *flags, cudaStream_t s, Overlap *ov) {
    if (open_faces(g)) return launch_faces_t<L, S, PSC>(fin, fout, g, ph, tl, pd, flags, s);
    if constexpr (sizeof(S) == 2) {
        return launch_collide_stream16<L, S, PSC>(fin, fout, g, ph, tl, pd, flags, s, ov);
    } else {
        // The adjoint's objective is one number, a sum over cells that may cancel to next to nothing
        // (128^3 with 200 spheres: 10 or 0.003 out of terms that add up to 200), so another order of
        // FP32 roundings in the state shows in its fourth digit although it is no less exact. Its
        // steps keep the order they had: 5.80 ms for 20 steps with gradient where k_step takes 5.41.
        if constexpr (sizeof(S) == 4 && PSC == 0) {
            if (tl.keep) return launch_collide_stream16<L, S, PSC>(fin, fout, g, ph, tl, pd, flags, s, ov);
        }
        // pairs in one access: every row of every direction starts on a pair boundary
        const bool vec = g.n[0] % 2 == 0 && ((uintptr_t)fin | (uintptr_t)fout) % (2 * sizeof(S)) == 0;
        if constexpr (L::D == 3 && sizeof(S) == 4) {
            if (g.wide)
                return vec ? launch_collide_stream_t<D3Q19w, S, PSC, true>(fin, fout, g, ph, tl, pd, flags, s, ov)
                           : launch_collide_stream_t<D3Q19w, S, PSC, false>(fin, fout, g, ph, tl, pd, flags, s, ov);
        }
        return vec ? launch_collide_stream_t<L, S, PSC, true>(fin, fout, g, ph, tl, pd, flags, s, ov)
                   : launch_collide_stream_t<L, S, PSC, false>(fin, fout, g, ph, tl, pd, flags, s, ov);
    }
}

template <typename S>
cudaError_t launch_collide_stream_storage(int lattice, const void *fin, void *fout, const Geom &g,
                                          const Phys &ph, const Tiles &tl, const Parts &pd,
                                          int *flags, cudaStream_t s, Overlap *ov) {
    if (lattice == 9) {
        return ph.psc == 0 ? launch_collide_stream_l<D2Q9, S, 0>(fin, fout, g, ph, tl, pd, flags, s, ov)
                           : launch_collide_stream_l<D2Q9, S, 1>(fin, fout, g, ph, tl, pd, flags, s, ov);
    }
    return ph.psc == 0 ? launch_collide_stream_l<D3Q19, S, 0>(fin, fout, g, ph, tl, pd, flags, s, ov)
                       : launch_collide_stream_l<D3Q19, S, 1>(fin, fout, g, ph, tl, pd, flags, s, ov);
}

template <class L, typename S>
cudaError_t launch_macro_t(const S *fin, double *rho, double *u, const Geom &g, const Phys &ph, cudaStream_t s) {
    auto kern = open_faces(g) ? k_macro<L, S, true> : k_macro<L, S, false>;
    const PhysT<typename Store<S>::T> pt = make_phys<typename Store<S>::T>(ph, L::Q);
    kern<<<dim3((unsigned)g.nt[0] * (unsigned)g.nt[1], 1, g.nt[2]), kThreads, 0, s>>>(fin, g, pt, (double)pt.F[0], (double)pt.F[1],
                                                             (double)pt.F[2], rho, u);
    return cudaGetLastError();
}

template <typename S>
cudaError_t launch_gather_storage(int lattice, const void *fin, double *f_out, double *rho,
                                  double *u, const Geom &g, const Phys &ph, cudaStream_t s) {
    using T = typename Store<S>::T;
    if (rho || u) {
        cudaError_t e = lattice == 9 ? launch_macro_t<D2Q9, S>((const S *)fin, rho, u, g, ph, s) : cudaSuccess;
        if (lattice != 9) {
            if constexpr (sizeof(S) == 4) {
                e = g.wide ? launch_macro_t<D3Q19w, S>((const S *)fin, rho, u, g, ph, s)
                           : launch_macro_t<D3Q19, S>((const S *)fin, rho, u, g, ph, s);
            } else {
                e = launch_macro_t<D3Q19, S>((const S *)fin, rho, u, g, ph, s);
            }
        }
        if (e != cudaSuccess || !f_out) return e;
    }
    const int threads = 256;
    const unsigned blocks = (unsigned)((g.ncell + threads - 1) / threads);
    if (lattice == 9) k_gather<D2Q9, S><<<blocks, threads, 0, s>>>((const S *)fin, g, make_phys<T>(ph, 9), f_out);
    else k_gather<D3Q19, S><<<blocks, threads, 0, s>>>((const S *)fin, g, make_phys<T>(ph, 19), f_out);
    return cudaGetLastError();
}

template <typename S>
cudaError_t launch_set_storage(int lattice, const double *f, void *fout, const Geom &g,
                               const Phys &ph, cudaStream_t s) {
    using T = typename Store<S>::T;
    const int threads = 256;
    const unsigned blocks = (unsigned)((g.ncell + threads - 1) / threads);
    if (lattice == 9) k_set<D2Q9, S><<<blocks, threads, 0, s>>>(f, (S *)fout, g, make_phys<T>(ph, 9));
    else k_set<D3Q19, S><<<blocks, threads, 0, s>>>(f, (S *)fout, g, make_phys<T>(ph, 19));
    return cudaGetLastError();
}

}  // namespace psc
