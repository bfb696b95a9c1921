// psc_pair.cuh -- the collide-stream step of lattices stored in FP32 and FP64 (included by
// psc_kernels.cuh inside namespace psc, after the shared helpers; 16 bits: psc_pair16.cuh).
//
// A warp works alone on 64 cells of a lattice tile at a time: two neighbouring rows of a tile 32
// wide (2D: rows 2k and 2k + 1; 3D: row k at both z), one per half warp, or one row of a tile 64
// wide (D3Q19w). Each lane owns two x-neighbours. Per 64 cells the warp
//   queues the pull of the populations (Eq. 1, 6);
//   tests the tile's candidate particles against its rows (one lane per candidate, ballot) and
//     visits those that can reach them for the solid fractions (Table 1, Eq. 15-18) and, for
//     moving particles, the u_s moments of the collision, while the populations are in flight;
//   forms the moments (Eq. 5), the weights (Eq. 9, 13), collides (Eq. 2-4, 10, 12) and stores;
//   visits the candidates again for force and torque (Eq. 14), sums them over the warp and
//     adds the sums with one FP64 atomic per component.
// The arithmetic runs on pairs (cell a, cell b = a + 1 in x); in FP32 a pair is one packed
// register pair and one FFMA2 / FADD2 / FMUL2 instruction does both cells.
//
// Why this shape. The step is bound by DRAM where tiles hold no particles and by instruction
// issue and latency where they do. With one cell per lane and row, forming 64-bit addresses was
// 45 % of the instructions; a pair of x-neighbours needs one address per direction (both values
// in one access where e_x = 0 and in every store, two loads at fixed offsets where e_x != 0). The
// memory system takes 55 to 65 G line requests a second whatever their size, so rows of 64
// bytes (32 cells of 16 bits) cost what lines of 128 do: a plain copy of 19 planes of 256^3
// 16-bit values by such rows takes 350 us, of 32-bit values 376 us; hence rows of 64 cells
// in 3D. Warps share nothing (no block barrier), so plain-fluid and particle rows interleave
// freely. Collide-stream kernels of a step, before (two rows of 32 cells, one cell per lane and
// row, blocks with a barrier per tile) and now, FP32: 256^3 with 2000 spheres 562 -> 421 us, 128^3
// with 200 spheres 79 -> 62, 2048^2 with 5000 discs in a band 69 -> 63, 777 x 453 with 500 discs
// 20.3 -> 15.6 (the state read and written once takes 376, 47, 44 and 3.7 us).
// Measured slower and not kept: rows copied one unit ahead into shared memory by cp.async (the
// shared memory comes out of the L1 that loads in flight need: with 200 KB of it a plain copy
// takes 478 us instead of 371); prefetching the next rows into L2 (30 % slower: as many requests
// again); a fixed stride over the tiles instead of counters (1.3 to 1.5 times as long).

constexpr int kPThreads = 128;
constexpr int kPWarps = kPThreads / 32;

// Pairs of the compute type: FP32 on the packed sm_100 instructions, FP64 as two scalars (rounded
// operations, not contracted, so that every instantiation rounds alike).
template <typename T> struct Pr;
template <> struct Pr<float> {
    using V = float2;
    static __device__ __forceinline__ V mk(float a, float b) { return make_float2(a, b); }
    static __device__ __forceinline__ V sp(float a) { return make_float2(a, a); }
    static __device__ __forceinline__ V add(V x, V y) { return __fadd2_rn(x, y); }
    static __device__ __forceinline__ V sub(V x, V y) { return __fadd2_rn(x, make_float2(-y.x, -y.y)); }
    static __device__ __forceinline__ V mul(V x, V y) { return __fmul2_rn(x, y); }
    static __device__ __forceinline__ V fma(V x, V y, V z) { return __ffma2_rn(x, y, z); }
};
template <> struct Pr<double> {
    using V = double2;
    static __device__ __forceinline__ V mk(double a, double b) { return make_double2(a, b); }
    static __device__ __forceinline__ V sp(double a) { return make_double2(a, a); }
    static __device__ __forceinline__ V add(V x, V y) { return make_double2(__dadd_rn(x.x, y.x), __dadd_rn(x.y, y.y)); }
    static __device__ __forceinline__ V sub(V x, V y) { return make_double2(__dsub_rn(x.x, y.x), __dsub_rn(x.y, y.y)); }
    static __device__ __forceinline__ V mul(V x, V y) { return make_double2(__dmul_rn(x.x, y.x), __dmul_rn(x.y, y.y)); }
    static __device__ __forceinline__ V fma(V x, V y, V z) {
        return make_double2(__fma_rn(x.x, y.x, z.x), __fma_rn(x.y, y.y, z.y));
    }
};

// num / den for normal den. FP32: the hardware's approximate reciprocal and one residual
// correction of the quotient (Markstein, "Computation of elementary functions on the IBM
// RISC System/6000", 1990): within 0.500001 ulp of the quotient for reciprocals up to two ulp off,
// which is the correctly rounded one but for one in 10^5 (emulated over the step's operands).
__device__ __forceinline__ float2 quot(const float2 num, const float2 den) {
    using P = Pr<float>;
    const float2 r = make_float2(__fdividef(1.0f, den.x), __fdividef(1.0f, den.y));
    const float2 q = P::mul(num, r);
    return P::fma(P::fma(make_float2(-q.x, -q.y), den, num), r, q);
}
__device__ __forceinline__ double2 quot(const double2 num, const double2 den) {
    return make_double2(num.x / den.x, num.y / den.y);
}

// One row of a pair's cells.
struct PairPos {
    int x, y, z;
    bool actA, actB;      // cells this context updates (b only where a)
};

// Where a step reads and writes each direction: plane i of the input shifted by the y and z
// components of its pull (x is the lane's), plane i of the output. Formed on the host: in the
// kernel each address is then one 64-bit sum with a constant, where the products and sums
// of plane and row strides took four times as many instructions.
template <class L, typename S> struct Dirs {
    const S *in[L::Q];
    S *out[L::Q];
    Dirs(const void *fin, void *fout, const Geom &g) {
        for (int i = 0; i < L::Q; ++i) {
            const long long o = i * g.ncell, r = L::ey(i) * (long long)g.n[0] + L::ez(i) * (long long)g.n[0] * g.n[1];
            in[i] = reinterpret_cast<const S *>(reinterpret_cast<intptr_t>(fin) + (o - r) * (long long)sizeof(S));
            out[i] = reinterpret_cast<S *>(reinterpret_cast<intptr_t>(fout) + o * (long long)sizeof(S));
        }
    }
};
// element k of direction i's plane (a pull's source, an output), k tested against the lattice
// in the bounds-checked build
template <class L, typename S>
__device__ __forceinline__ const S *src_at(const Dirs<L, S> &f, const Geom &g, const int i, const long long k) {
#ifdef PSC_CHECKED
    const long long o = (long long)i * g.ncell - (L::ey(i) * (long long)g.n[0] + L::ez(i) * (long long)g.n[0] * g.n[1]);
    return f.in[0] + PSC_IDX(k + o, L::Q * g.ncell, CHK_POP);
#else
    (void)g;
    return f.in[i] + k;
#endif
}
template <class L, typename S>
__device__ __forceinline__ S *dst_at(const Dirs<L, S> &f, const Geom &g, const int i, const long long k) {
#ifdef PSC_CHECKED
    return f.out[0] + PSC_IDX(k + (long long)i * g.ncell, L::Q * g.ncell, CHK_POP);
#else
    (void)g;
    return f.out[i] + k;
#endif
}

// Two x-neighbours, in one access (VEC: the rows start on a pair boundary) or two.
template <typename S, bool VEC>
__device__ __forceinline__ void ld_pair(const S *p, typename Store<S>::T &a, typename Store<S>::T &b) {
    if (!VEC) {
        a = Store<S>::ldr(p, 0);
        b = Store<S>::ldr(p, 1);
    } else if constexpr (sizeof(S) == 8) {
        const double2 v = *reinterpret_cast<const double2 *>(p);
        a = v.x; b = v.y;
    } else {
        const float2 v = *reinterpret_cast<const float2 *>(p);
        a = v.x; b = v.y;
    }
}
// Stores of a pair: together where rows start on a pair boundary.
template <typename S, bool VEC>
__device__ __forceinline__ void st_pair(S *p, const typename Store<S>::T a, const typename Store<S>::T b, const bool actB) {
    if (!VEC) {
        Store<S>::str(p, 0, a);
        if (actB) Store<S>::str(p, 1, b);
    } else if constexpr (sizeof(S) == 8) {
        *reinterpret_cast<double2 *>(p) = make_double2(a, b);
    } else {
        *reinterpret_cast<float2 *>(p) = make_float2(a, b);
    }
}

// Where a warp's 64 cells lie: its tile's origin and which of the tile's four such units, two rows
// (2D: rows 2k and 2k + 1; 3D: row k at both z) or, in tiles 64 wide (3D), row k / 2 at z = k % 2.
template <class L> struct UnitPos {
    static constexpr bool kWide = L::TX == 64;
    int x0, y0, z0, k;
    // in the tile, of row r (0 or 1; the same where wide)
    __device__ __forceinline__ int ry(const int r) const { return L::D == 2 ? 2 * k + r : (kWide ? k >> 1 : k); }
    __device__ __forceinline__ int rz(const int r) const { return L::D == 2 ? 0 : (kWide ? k & 1 : r); }
    __device__ __forceinline__ int y(const int r) const { return y0 + ry(r); }
    __device__ __forceinline__ int z(const int r) const { return z0 + rz(r); }
};
constexpr int kUnits = 4;        // per tile

// Rows whose pull stays inside the lattice but for a wrap of pairs in x: every neighbour row
// exists, and the pairs are clear of the x faces or on a periodic axis where none straddles the end.
template <class L>
__device__ __forceinline__ bool unit_inner(const Geom &g, const UnitPos<L> &u) {
    const bool x = (g.periodic[0] || (u.x0 >= 1 && u.x0 + L::TX < g.n[0])) && (!(g.n[0] & 1) || u.x0 + L::TX < g.n[0]);
    return x && u.y(0) >= 1 && u.y(1) + 1 < g.n[1] && (L::D == 2 || (u.z(0) >= 1 && u.z(1) + 1 < g.n[2]));
}

// Pull of a pair of inner rows (see unit_inner). One address per direction; where e_x != 0 the
// value beyond the pair comes by its own (wrapped) place. Lanes past an even row's end read its
// last pair.
template <class L, typename S, bool VEC>
__device__ __forceinline__ void pull_inner(const Dirs<L, S> &f, const Geom &g, const PairPos &c,
                                           typename Store<S>::T *da, typename Store<S>::T *db) {
    const int x = min(c.x, g.n[0] - 2);
    const long long p = x + (long long)g.n[0] * (c.y + (long long)g.n[1] * c.z);
    const long long pm = p + (x == 0 ? g.n[0] - 1 : -1), pp = p + (x + 2 == g.n[0] ? 2 - g.n[0] : 2);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const S *const q = src_at<L, S>(f, g, i, p);
        if (L::ex(i) == 0) {
            ld_pair<S, VEC>(q, da[i], db[i]);
        } else if (L::ex(i) > 0) {
            da[i] = Store<S>::ldr(src_at<L, S>(f, g, i, pm), 0);
            db[i] = Store<S>::ldr(q, 0);
        } else {
            da[i] = Store<S>::ldr(q, 1);
            db[i] = Store<S>::ldr(src_at<L, S>(f, g, i, pp), 0);
        }
    }
}

// Pull of a pair anywhere in a lattice with periodic and wall faces.
template <class L, typename S>
__device__ __forceinline__ void pull_edge(const S *__restrict__ fin, const Geom &g, const PairPos &c,
                                          typename Store<S>::T *da, typename Store<S>::T *db) {
    const long long cell = c.x + (long long)g.n[0] * (c.y + (long long)g.n[1] * c.z);
    pull_q<L, S, true>(fin, g, c.x, c.y, c.z, cell, false, c.actA, make_float2(1.0f, 1.0f), da);
    pull_q<L, S, true>(fin, g, c.x + 1, c.y, c.z, cell + 1, false, c.actB, make_float2(1.0f, 1.0f), db);
}

// Solid fractions kept per lane between the two visits.
constexpr int kSlots = 4;

// Solid fractions of a candidate at the pair: x-distance dx of cell a (b: dx + 1), squared
// distance c2 in the other axes (Table 1 Steps 2-4, D = distance - r; see shell_eps).
__device__ __forceinline__ float2 shell_pair(const float2 dx, const float c2, const float r, const float fr, const float h) {
    using P = Pr<float>;
    const float2 d2 = P::fma(dx, dx, P::sp(c2));
    float2 q;      // rsqrt of a normal number
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(q.x) : "f"(fmaxf(d2.x, 1e-30f)));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(q.y) : "f"(fmaxf(d2.y, 1e-30f)));
    const float2 D = P::add(P::mul(d2, q), P::sp(-r));
    float ea = __saturatef(fr - D.x), eb = __saturatef(fr - D.y);
    ea = D.x <= -h ? 1.0f : (D.x < h ? ea : 0.0f);
    eb = D.y <= -h ? 1.0f : (D.y < h ? eb : 0.0f);
    return make_float2(ea, eb);
}
__device__ __forceinline__ double2 shell_pair(const double2 dx, const double c2, const double r, const double fr,
                                              const double h) {
    return make_double2(shell_eps<double>(dx.x * dx.x + c2, r, fr, h), shell_eps<double>(dx.y * dx.y + c2, r, fr, h));
}

// Collision of a pair (Eq. 2-4, 10, 12), each direction as
//   out_i = a d_i + B d_-i + w_i (E_i + O_i),   E_i = K + e.A.e,  O_i = e.q,
//   a = 1 - omega(1-B) - B,  q = 3 (omega(1-B) + B) rho u + 3 rho c_B m + 3 cg F,
//   A = 4.5 rho (omega(1-B) - B) u u^T + 4.5 rho c_B M + 4.5 cg (F u^T + u F^T),
//   K = omega(1-B) drho - tr(A) / 3,  cg = (1-B)(1 - 1/(2 tau)),
// m, M the u_s moments before the normalisation c_B of Eq. 13. E is common to a direction and
// its opposite and O changes sign, so a pair of opposite directions costs one of each; K, A and
// q carry the weight of a diagonal direction (1/36). Without solid cells
// (B = 0) the same operations with fewer terms: the results do not depend on SOLID.
// q is the cell's momentum rho u = j + F/2 times 3/36, which is no FP32 number: it is applied
// as a rounded constant and its remainder, since a constant 3e-8 off would add as much to every
// cell's momentum in every step (drag of a sphere over 20 steps: twice the error).
template <class L, typename S, bool SOLID, bool VEC>
__device__ __forceinline__ void collide_store(const Dirs<L, S> &f, const Geom &g, const PhysT<typename Store<S>::T> &ph,
                                              const PairPos &c, typename Store<S>::T *da,
                                              typename Store<S>::T *db, const typename Pr<typename Store<S>::T>::V drho,
                                              const typename Pr<typename Store<S>::T>::V rho,
                                              const typename Pr<typename Store<S>::T>::V *u,
                                              const typename Pr<typename Store<S>::T>::V *mom,
                                              const typename Pr<typename Store<S>::T>::V Bn,
                                              const typename Pr<typename Store<S>::T>::V cB,
                                              const typename Pr<typename Store<S>::T>::V *m,
                                              const typename Pr<typename Store<S>::T>::V *M) {
    using T = typename Store<S>::T;
    using P = Pr<T>;
    using V = typename P::V;
    constexpr int D = L::D;
    constexpr T kAxis = (D == 2) ? (T)4 : (T)2, kRest = (D == 2) ? (T)16 : (T)12;   // weights over the diagonal's
    const T ws = (T)(1.0 / 36.0);
    const V one = P::sp((T)1);
    const V omB = SOLID ? P::sub(one, Bn) : one;
    const V oo = SOLID ? P::mul(omB, P::sp(ph.omega)) : P::sp(ph.omega);
    const V rest = P::sub(one, oo), a = SOLID ? P::sub(rest, Bn) : rest;
    const V r45 = P::mul(rho, P::sp((T)4.5 * ws)), r3 = P::mul(rho, P::sp((T)3 * ws));
    const V al = P::mul(r45, SOLID ? P::sub(oo, Bn) : oo);
    const V be = SOLID ? P::add(oo, Bn) : oo;
    const T c12 = ph.c12[0], c12r = ph.c12[1];      // 1 / 12 and its remainder
    // (a product that is added to later is formed as a fused operation with this run-time zero:
    // the compiler fuses packed products and sums, and differently in each instantiation)
    const V none = P::sp(ph.none);
    V q[3], A[3], X[3];       // A: diagonal; X: twice the off-diagonal xy, xz, yz
    {
        V t[3], gF[3];        // t = 4.5 cg F + al u
#pragma unroll
        for (int k = 0; k < D; ++k) {
            const V cg = SOLID ? P::mul(omB, P::sp(ph.guo)) : P::sp(ph.guo);
            gF[k] = P::fma(cg, P::sp((T)4.5 * ws * ph.F[k]), none);
            t[k] = P::fma(al, u[k], gF[k]);
            const V bm = P::mul(be, mom[k]);
            q[k] = P::fma(bm, P::sp(c12), P::fma(bm, P::sp(c12r), P::mul(cg, P::sp((T)3 * ws * ph.F[k]))));
            A[k] = P::fma(u[k], P::add(t[k], gF[k]), none);
        }
        X[0] = P::fma(u[0], t[1], P::mul(gF[0], u[1]));
        if (D == 3) {
            X[1] = P::fma(u[0], t[2], P::mul(gF[0], u[2]));
            X[2] = P::fma(u[1], t[2], P::mul(gF[1], u[2]));
        }
    }
    if (SOLID) {
        const V b45 = P::mul(r45, cB), b3 = P::mul(r3, cB);
#pragma unroll
        for (int k = 0; k < D; ++k) {
            q[k] = P::fma(b3, m[k], q[k]);
            A[k] = P::fma(b45, M[k], A[k]);
        }
        X[0] = P::fma(b45, M[3], X[0]);
        if (D == 3) {
            X[1] = P::fma(b45, M[4], X[1]);
            X[2] = P::fma(b45, M[5], X[2]);
        }
    }
    const V tr = (D == 3) ? P::add(A[0], P::add(A[1], A[2])) : P::add(A[0], A[1]);
    const V K = P::fma(tr, P::sp((T)(-1.0 / 3.0)), P::mul(P::mul(oo, P::sp(ws)), drho));
    auto put = [&](const int i, const V v) { da[i] = v.x; db[i] = v.y; };      // in place
    auto d = [&](const int i) { return P::mk(da[i], db[i]); };
    // directions i and i + 1 = -i with even and odd parts E, O at f times the diagonal weight
    auto both = [&](const int i, const V E, const V O, const bool axis) {
        const V s0 = P::add(E, O), s1 = P::sub(E, O);
        const V d0 = d(i), d1 = d(i + 1);
        V t0 = axis ? P::mul(s0, P::sp(kAxis)) : s0, t1 = axis ? P::mul(s1, P::sp(kAxis)) : s1;
        if (SOLID) { t0 = P::fma(Bn, d1, t0); t1 = P::fma(Bn, d0, t1); }
        put(i, P::fma(a, d0, t0));
        put(i + 1, P::fma(a, d1, t1));
    };
    put(0, P::fma(rest, d(0), P::mul(K, P::sp(kRest))));
    V E[3];
#pragma unroll
    for (int k = 0; k < D; ++k) {
        E[k] = P::add(K, A[k]);
        both(1 + 2 * k, E[k], q[k], true);
    }
    // diagonal directions in the plane of axes (j, k): e = (1, 1) and (1, -1)
    auto plane = [&](const int i, const int j, const int k, const V x) {
        const V E0 = P::add(E[j], A[k]);
        const V x2 = P::add(x, x);
        both(i, P::add(E0, x2), P::add(q[j], q[k]), false);
        both(i + 2, P::sub(E0, x2), P::sub(q[j], q[k]), false);
    };
    if (D == 2) {
        plane(5, 0, 1, X[0]);
    } else {
        plane(7, 0, 1, X[0]);
        plane(11, 0, 2, X[1]);
        plane(15, 1, 2, X[2]);
    }
    if (c.actA) {       // b is active only where a is
        const long long k = c.x + (long long)g.n[0] * (c.y + (long long)g.n[1] * c.z);
#pragma unroll
        for (int i = 0; i < L::Q; ++i) st_pair<S, VEC>(dst_at<L, S>(f, g, i, k), da[i], db[i], c.actB);
    }
}

// The arm from candidate q (position, radius) to the pair at c (cell a) on lattices with periodic
// axes too short for the tile's own image of the candidate to be the nearest for every cell. What
// the difference over up to a period loses in rounding is added back to the short arm.
template <typename T> struct Arm {
    typename Pr<T>::V dx;
    T dy, dz;
};
template <class L, typename T>
__device__ __noinline__ Arm<T> near_image(const Geom &g, const T h, const Vec4<T> q, const T cx, const T cy, const T cz) {
    const int ext[3] = {L::TX, L::TY, L::TZ};
    auto image = [&](const T c, const T p, const int a) {
        const T n = (T)g.n[a], v = c - p;
        if (!g.wrap_img[a] || !(n < (T)(ext[a] + 2) + (T)2 * (q.w + h))) return v;
        const T b = v - c, lost = (c - (v - b)) - (p + b);
        return (v - n * rint_t(v / n)) + lost;
    };
    Arm<T> r;
    r.dx = Pr<T>::mk(image(cx, q.x, 0), image(cx + (T)1, q.x, 0));
    r.dy = image(cy, q.y, 1);
    r.dz = (L::D == 3) ? image(cz, q.z, 2) : (T)0;
    return r;
}

// A warp's 64 cells, with the tile's cnt candidate records (SOLID).
template <class L, typename S, int PSC, bool SOLID, bool VEC>
__device__ __forceinline__ void unit_step(const UnitPos<L> &up, const int cnt,
                                          const typename Store<S>::T *__restrict__ recs,
                                          const Dirs<L, S> &f, const Geom &g, const PhysT<typename Store<S>::T> &ph,
                                          const Parts &pd, int *flags, typename Pr<typename Store<S>::T>::V *slots) {
    using T = typename Store<S>::T;
    using P = Pr<T>;
    using V = typename P::V;
    constexpr int Q = L::Q, D = L::D;
    constexpr bool WIDE = UnitPos<L>::kWide;
    const int lane = threadIdx.x & 31;
    const int cxi = WIDE ? 2 * lane : 2 * (lane & 15), row = lane >> 4;    // the pair's first cell, row
    PairPos c;
    c.x = up.x0 + cxi; c.y = up.y(row); c.z = up.z(row);
    {
        const bool in = (D == 2) ? (unsigned)(c.y - g.act0) < (unsigned)(g.act1 - g.act0)
                                 : (c.y < g.n[1] && (unsigned)(c.z - g.act0) < (unsigned)(g.act1 - g.act0));
        c.actA = in && c.x < g.n[0];
        c.actB = in && c.x + 1 < g.n[0];
    }
    T da[Q], db[Q];
    if (unit_inner<L>(g, up)) pull_inner<L, S, VEC>(f, g, c, da, db);
    else pull_edge<L, S>(f.in[0], g, c, da, db);
    const V zero = P::sp((T)0);
    V seps = zero, m[3] = {zero, zero, zero}, M[6] = {zero, zero, zero, zero, zero, zero};
    // tile-relative: the two rows (the same where wide), the lane's own
    const T fy0 = (T)up.ry(0), fy1 = (T)up.ry(1), fz0 = (T)up.rz(0), fz1 = (T)up.rz(1);
    const T cx = (T)(cxi - L::REC_X), cy = (WIDE || row == 0) ? fy0 : fy1, cz = (WIDE || row == 0) ? fz0 : fz1;
    const bool wrapped = g.wrap_img[0] || g.wrap_img[1] || g.wrap_img[2];

    // ---- candidates that can reach the rows
    unsigned wmask = 0u;
    if (SOLID && cnt > 0) {
        bool rel = false;
        if (lane < cnt) {
            const Vec4<T> q = ld4<T>(recs + lane * RW);
            const T xmax = (T)(min(L::TX, g.n[0] - up.x0) - 1);
            rel = row_hits<L, T>(g, q.x + (T)L::REC_X, q.y, q.z, q.w + ph.h, fy0, fz0, xmax);
            if (!WIDE) rel = rel || row_hits<L, T>(g, q.x + (T)L::REC_X, q.y, q.z, q.w + ph.h, fy1, fz1, xmax);
        }
        wmask = __ballot_sync(kFull, rel);
    }
    // arm from candidate q to the pair (x of cell a and b; y and z are common)
    auto arm = [&](const Vec4<T> &q, V &dx, T &dy, T &dz) {
        const T dxa = cx - q.x;
        dy = cy - q.y;
        dz = (D == 3) ? cz - q.z : (T)0;
        dx = P::mk(dxa, cx + (T)1 - q.x);
        if (wrapped) {
            const Arm<T> n = near_image<L, T>(g, ph.h, q, cx, cy, cz);
            dx = n.dx; dy = n.dy; dz = n.dz;
        }
    };
    auto fraction = [&](const Vec4<T> &q, const T fr, const V dx, const T dy, const T dz) {
        V e = shell_pair(dx, dy * dy + dz * dz, q.w, fr, ph.h);
        if (!c.actA) e.x = (T)0;
        if (!c.actB) e.y = (T)0;
        return e;
    };
    // u_s = U + Omega x (x_n - X_p); U in y, z, w of v
    auto us_at = [&](const Vec4<T> &v, const Vec4<T> &o, const V dx, const T dy, const T dz, V *us) {
        us[0] = P::fma(P::sp(o.y), P::sp(dz), P::fma(P::sp(-o.z), P::sp(dy), P::sp(v.y)));
        us[1] = P::fma(P::sp(o.z), dx, P::fma(P::sp(-o.x), P::sp(dz), P::sp(v.z)));
        us[2] = (D == 3) ? P::fma(P::sp(o.x), P::sp(dy), P::fma(P::sp(-o.y), dx, P::sp(v.w))) : zero;
    };

    // ---- solid fractions and u_s moments
    V *const slot = slots + lane;
    {
        unsigned mk = wmask;
        for (int js = 0; mk != 0u; ++js) {
            const int k = __ffs(mk) - 1;
            mk &= mk - 1u;
            const T *rk = recs + k * RW;
            const Vec4<T> q = ld4<T>(rk), v = ld4<T>(rk + 4);
            {
                V dx;
                T dy, dz;
                arm(q, dx, dy, dz);
                const V e = fraction(q, fabs(v.x), dx, dy, dz);
                if (js < kSlots) slot[32 * js] = e;
                // modified scheme weights by eps_s (normalised below); original by B(eps_s)
                const V wgt = (PSC == 0) ? e : quot(P::mul(e, P::sp(ph.tmh)), P::add(P::sub(P::sp((T)1), e), P::sp(ph.tmh)));
                seps = P::add(seps, wgt);
                if (v.x < (T)0) {          // a moving particle
                    const Vec4<T> o = ld4<T>(rk + 8);
                    V us[3], w[3];
                    us_at(v, o, dx, dy, dz, us);
#pragma unroll
                    for (int a = 0; a < D; ++a) {
                        w[a] = P::mul(wgt, us[a]);
                        m[a] = P::add(m[a], w[a]);
                        M[a] = P::fma(w[a], us[a], M[a]);
                    }
                    M[3] = P::fma(w[0], us[1], M[3]);
                    if (D == 3) {
                        M[4] = P::fma(w[0], us[2], M[4]);
                        M[5] = P::fma(w[1], us[2], M[5]);
                    }
                }
            }
        }
    }

    V J[3], rho, Bn, cB;
    {
        // ---- moments (Eq. 5)
        auto d = [&](const int i) { return P::mk(da[i], db[i]); };
        V drho = d(0), j[3] = {zero, zero, zero};
#pragma unroll
        for (int i = 1; i < Q; ++i) drho = P::add(drho, d(i));
        {
            bool first[3] = {true, true, true};
#pragma unroll
            for (int i = 1; i < Q; i += 2) {      // d_i - d_-i, shared by the axes it enters
                const V o = P::sub(d(i), d(i + 1));
                const int e[3] = {L::ex(i), L::ey(i), L::ez(i)};
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    if (!e[k]) continue;
                    if (first[k]) { j[k] = e[k] > 0 ? o : P::sub(zero, o); first[k] = false; }
                    else j[k] = e[k] > 0 ? P::add(j[k], o) : P::sub(j[k], o);
                }
            }
        }
        rho = P::add(P::sp((T)1), drho);
        const V irho = quot(P::sp((T)1), rho);
        V u[3], mom[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            J[k] = j[k];
            mom[k] = P::add(j[k], P::sp((T)0.5 * ph.F[k]));
            u[k] = P::mul(mom[k], irho);
        }
        if ((c.actA && !(rho.x > (T)0)) || (c.actB && !(rho.y > (T)0))) atomicOr(flags, 1);

        // ---- weights (Table 1 Step 5, Eq. 9, 13): eps_n = min(1, sum eps), B_n by Eq. 9 at
        //      eps_n, B_{n,s} = c_B eps_s; original scheme: B_n = sum_s B(eps_s) (Eq. 8), c_B = 1
        Bn = cB = zero;
        if (SOLID && wmask != 0u) {
            if (PSC == 0) {
                const bool fa = seps.x < (T)1, fb = seps.y < (T)1;
                const V num = P::mk(fa ? ph.tmh : (T)1, fb ? ph.tmh : (T)1);
                const V den = P::mk(fa ? ((T)1 - seps.x) + ph.tmh : seps.x, fb ? ((T)1 - seps.y) + ph.tmh : seps.y);
                cB = quot(num, den);
                Bn = P::mul(seps, cB);
                if (!fa) Bn.x = (T)1;
                if (!fb) Bn.y = (T)1;
            } else {
                Bn = seps;
                cB = P::sp((T)1);
            }
        }
        collide_store<L, S, SOLID, VEC>(f, g, ph, c, da, db, drho, rho, u, mom, Bn, cB, m, M);
    }
    if (!SOLID) return;

    // ---- force and torque (Eq. 14; Eq. 11 original): F_p -= B (rho u_s + F/2 - j),
    //      T_p -= (x_n - X_p) x the same, over the lane's cells, then over the warp
    constexpr int NCP = (D == 2) ? 4 : 8, NC = (D == 2) ? 3 : 6;
    for (int js = 0; wmask != 0u; ++js) {
        const int k = __ffs(wmask) - 1;
        wmask &= wmask - 1u;
        const T *rk = recs + k * RW;
        const Vec4<T> q = ld4<T>(rk), v = ld4<T>(rk + 4), o = ld4<T>(rk + 8);
        T t[NCP];
#pragma unroll
        for (int a = 0; a < NCP; ++a) t[a] = (T)0;
        bool any = false;
        {
            V dx;
            T dy, dz;
            arm(q, dx, dy, dz);
            const V e = js < kSlots ? slot[32 * js] : fraction(q, fabs(v.x), dx, dy, dz);
            any |= e.x > (T)0 || e.y > (T)0;
            const V w = (PSC == 0) ? P::mul(cB, e) : P::mk(e.x > (T)0 ? Bn.x : (T)0, e.y > (T)0 ? Bn.y : (T)0);
            V P0[3];       // F/2 - j, the fluid part of the momentum exchange, and rho u_s
#pragma unroll
            for (int a = 0; a < D; ++a) P0[a] = P::sub(P::sp((T)0.5 * ph.F[a]), J[a]);
            if (v.x < (T)0) {
                V us[3];
                us_at(v, o, dx, dy, dz, us);
#pragma unroll
                for (int a = 0; a < D; ++a) P0[a] = P::fma(rho, us[a], P0[a]);
            }
            T s[3] = {(T)0, (T)0, (T)0}, sx[3] = {(T)0, (T)0, (T)0};   // sums of dP and of dx dP over a, b
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const V dP = P::mul(w, P0[a]);
                s[a] = dP.x + dP.y;
                if (a > 0) sx[a] = dx.x * dP.x + dx.y * dP.y;
            }
            t[0] += s[0];
            t[1] += s[1];
            if (D == 2) {
                t[2] += sx[1] - dy * s[0];
            } else {
                t[2] += s[2];
                t[3] += dy * s[2] - dz * s[1];
                t[NCP - 4] += dz * s[0] - sx[2];
                t[NCP - 3] += sx[1] - dy * s[0];
            }
        }
        if (!__any_sync(kFull, any)) continue;
        const T tot = warp_sum_spread<NCP>(t, lane);
        const int cs = lane / (32 / NCP);
        if ((lane & (32 / NCP - 1)) == 0 && cs < NC && tot != (T)0) {
            const int pid = (int)PSC_IDX(bits_id(o.w), pd.n, CHK_PART);
            double *dst;
            if (D == 2) dst = (cs < 2) ? &pd.F[3 * pid + cs] : &pd.T[3 * pid + 2];
            else dst = (cs < 3) ? &pd.F[3 * pid + cs] : &pd.T[3 * pid + cs - 3];
            atomicAdd(dst, -(double)tot);
        }
    }
}

// Which lists of tiles a launch takes.
enum StepTiles {
    kParticleTiles = 1,    // the list of tiles with candidates
    kFluidTiles = 2,       // the list of tiles without
    kBothLists = 3         // those with candidates first
};

// First cell of a tile.
template <class L> __device__ __forceinline__ void unit_origin(const Geom &g, const unsigned tile, UnitPos<L> &u) {
    const unsigned t1 = tile / (unsigned)g.nt[0], tz = t1 / (unsigned)g.nt[1];
    u.x0 = (int)(tile - t1 * (unsigned)g.nt[0]) * L::TX;
    u.y0 = (int)(t1 - tz * (unsigned)g.nt[1]) * L::TY;
    u.z0 = (int)tz * L::TZ;
}

// One collide-stream step over the tiles of the lists `which`: persistent warps, an item being a
// tile or (shift > 0) one of 1 << shift equal parts of its units. Items go through work counters
// (they differ in cost, and so do SMs in their distance from memory), kCounters of them, a block's
// warps sharing one, since a single counter's atomics would take as long as the step of a 2D
// lattice. An item's number is fetched two items ahead of its turn, its tile one. The counters
// are cleared by an earlier kernel (k_clear): at the end of this one, the last fetch of a warp, which
// nothing waits for, might land after a clearing store of another. Tiles with more than kPairCap
// candidates are left to k_collide_overflow.
//
// Blocks per SM (registers): more or fewer measured slower (3D FP32, 256^3 with 2000 spheres: 5
// instead of 4 took 1.32 times as long, 3 on narrow tiles 1.06 times).
template <class L, typename S> __host__ __device__ constexpr int step_blocks() {
    return sizeof(S) == 8 ? 2 : (L::D == 2 ? 6 : 4);
}
template <class L, typename S, int PSC, bool SOLID, bool VEC>
__global__ void __launch_bounds__(kPThreads, (step_blocks<L, S>()))
k_step(const __grid_constant__ Dirs<L, S> f, const __grid_constant__ Geom g,
       const __grid_constant__ PhysT<typename Store<S>::T> ph, Tiles tl, Parts pd, int *flags, int *work, int which, int shift) {
    using T = typename Store<S>::T;
    using V = typename Pr<T>::V;
    __shared__ V s_slots[SOLID ? kPWarps * kSlots * 32 : 1];
    pdl_wait();
    pdl_launch();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned ntiles = (unsigned)g.nt[0] * (unsigned)g.nt[1] * (unsigned)g.nt[2];
    const unsigned np = (SOLID && (which & kParticleTiles)) ? (unsigned)tl.stats[4] : 0u;
    const unsigned nlist = np + ((which & kFluidTiles) ? (unsigned)tl.stats[5] : 0u);
    const long long nitem = (long long)nlist << shift;       // 1 << shift items a tile
    const int units = kUnits >> shift;
    const int groups = min(kCounters, (int)gridDim.x), group = blockIdx.x % groups;
    int *const counter = work + group * kCounterStride;
    auto fetch = [&]() { return lane == 0 ? atomicAdd(counter, 1) : 0; };       // lane 0's, not waited for
    auto number = [&](const int raw) { return (long long)__shfl_sync(kFull, raw, 0) * groups + group; };
    // the tile of an item (a load for lists)
    auto tile_of = [&](const long long it) {
        if (it >= nitem) return 0u;
        const unsigned ti = (unsigned)(it >> shift);
        return (unsigned)PSC_IDX(tl.order[ti < np ? ti : ntiles + (ti - np)], ntiles, CHK_TILE);
    };
    const T *const blocks = reinterpret_cast<const T *>(tl.blocks);
    const int limit = min(tl.cap, kPairCap);
    long long it = number(fetch());
    int raw = fetch();
    unsigned tile = tile_of(it);
    while (it < nitem) {
        const long long nx = number(raw);
        raw = fetch();
        const unsigned ntile = tile_of(nx);
        UnitPos<L> u;
        unit_origin<L>(g, tile, u);
        const int k0 = (int)(it & ((1 << shift) - 1)) * units;
        const int cnt = (SOLID && it < ((long long)np << shift)) ? tl.count[tile] : 0;
        const T *const recs = blocks + (size_t)tile * block_elems<T>(tl.cap) + head_elems<T>();
        if (cnt <= limit) {
#pragma unroll 1
            for (u.k = k0; u.k < k0 + units; ++u.k)
                unit_step<L, S, PSC, SOLID, VEC>(u, cnt, recs, f, g, ph, pd, flags,
                                                 s_slots + (SOLID ? warp * kSlots * 32 : 0));
        }
        it = nx; tile = ntile;
    }
}

// One step of a lattice without particles: no lists, so a unit per warp in the order of the blocks
// and no counters to share out. Bound by DRAM: 2048^2 FP32 47.6 us, 256^3 367 (the state once 44 and
// 376 at the copy's rate); warps that drew their units from counters took 54 and 381.
template <class L, typename S, bool VEC>
__global__ void __launch_bounds__(kPThreads, (step_blocks<L, S>()))
k_fluid(const __grid_constant__ Dirs<L, S> f, const __grid_constant__ Geom g,
        const __grid_constant__ PhysT<typename Store<S>::T> ph, int *flags) {
    pdl_wait();
    pdl_launch();
    const unsigned it = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    UnitPos<L> u;
    unit_origin<L>(g, it / kUnits, u);
    u.k = (int)(it % kUnits);
    unit_step<L, S, 0, false, VEC>(u, 0, nullptr, f, g, ph, Parts{}, flags, nullptr);
}
