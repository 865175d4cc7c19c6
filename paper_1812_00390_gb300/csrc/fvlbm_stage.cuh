// Templated CUDA kernels of one FVLBM stage (included by one translation unit
// per precision so that the build compiles them in parallel).
#pragma once

#include "fvlbm_device.cuh"
#include "fvlbm_internal.h"

namespace fvlbm {

template <typename T> __device__ __forceinline__ T inst_dt(const InstParam& p);
template <> __device__ __forceinline__ double inst_dt<double>(const InstParam& p) { return p.dt; }
template <> __device__ __forceinline__ float inst_dt<float>(const InstParam& p) { return p.dt_f; }
template <typename T> __device__ __forceinline__ T inst_inv_tau(const InstParam& p);
template <> __device__ __forceinline__ double inst_inv_tau<double>(const InstParam& p) { return p.inv_tau; }
template <> __device__ __forceinline__ float inst_inv_tau<float>(const InstParam& p) { return p.inv_tau_f; }

// ------------------------------------------------------------------ physics
// Ghost state of a boundary slot (Sec. 2.4.1): the stencil value of direction
// a minus the cell value is
//   wall      f^eq(rho, u_w) - f^eq(rho, u)                        Eq. (wallbc)
//   inlet     f^eq(rho*, u_inf) - f^eq(rho, u), rho* = rho_inf (external) or rho
//   outlet    0 (external) or f^eq(rho_inf, u) - f^eq(rho, u) (internal)
//   symmetry  f^eq(rho, u*) - f_a, u* = u mirrored in the face line
// i.e. f^eq(r, u_g) minus f^eq(rho, u) (or f_a for symmetry), with the ghost
// density / velocity (r, u_g) found once per slot.
template <typename T> struct Ghost {
    T r, ux, uy;
    bool zero;    // external outlet: no difference
    bool sym;     // symmetry: subtract f_a
    bool io;      // inlet / internal outlet: faces the cell flows out through are reconstructed
};

// Boundary constants in the arithmetic type (FP32: rounded on the host).
template <typename T> struct BcVal;
template <> struct BcVal<double> {
    static __device__ __forceinline__ double uwx(const BcParam& b) { return b.uwx; }
    static __device__ __forceinline__ double uwy(const BcParam& b) { return b.uwy; }
    static __device__ __forceinline__ double uix(const BcParam& b) { return b.uix; }
    static __device__ __forceinline__ double uiy(const BcParam& b) { return b.uiy; }
    template <bool DEV> static __device__ __forceinline__ double rho(const BcParam& b) { return rarg<double, DEV>(b.rho_inf); }
};
template <> struct BcVal<float> {
    static __device__ __forceinline__ float uwx(const BcParam& b) { return b.uwx_f; }
    static __device__ __forceinline__ float uwy(const BcParam& b) { return b.uwy_f; }
    static __device__ __forceinline__ float uix(const BcParam& b) { return b.uix_f; }
    static __device__ __forceinline__ float uiy(const BcParam& b) { return b.uiy_f; }
    template <bool DEV> static __device__ __forceinline__ float rho(const BcParam& b) { return DEV ? b.rdev_f : b.rho_f; }
};

template <typename T, bool DEV, typename NormalFn>
__device__ __forceinline__ Ghost<T> ghost_state(uint32_t kind, const BcParam& b, T rho, T ux, T uy, NormalFn normal) {
    Ghost<T> g{rho, ux, uy, false, false, false};
    if (kind == LK_WALL) {
        g.ux = BcVal<T>::uwx(b);
        g.uy = BcVal<T>::uwy(b);
    } else if (kind == LK_INLET) {
        if (b.external) g.r = BcVal<T>::template rho<DEV>(b);
        g.ux = BcVal<T>::uix(b);
        g.uy = BcVal<T>::uiy(b);
        g.io = true;
    } else if (kind == LK_OUTLET) {
        g.zero = true;
    } else if (kind == LK_PRESSURE) {
        g.r = BcVal<T>::template rho<DEV>(b);
        g.io = true;
    } else {   // symmetry: the face's unit normal is needed only here
        const typename Vec2<T>::type n = normal();
        const T inv = T(1) / sqrt(square(n.x, n.y));
        const T nhx = mul_rn(n.x, inv), nhy = mul_rn(n.y, inv);
        const T un2 = T(-2) * fma(ux, nhx, mul_rn(uy, nhy));
        g.ux = fma(un2, nhx, ux);
        g.uy = fma(un2, nhy, uy);
        g.sym = true;
    }
    return g;
}

// Stencil value minus cell value of direction a (fe = f^eq_a(rho, u)).
template <typename T, bool DEV>
__device__ __forceinline__ T ghost_delta(const Ghost<T>& g, int a, T fa, T fe) {
    if (g.zero) return T(0);
    return fma(feq_factor<T, DEV>(a, g.r), feq_value<T, DEV>(a, g.r, g.ux, g.uy), g.sym ? -fa : -fe);
}

__device__ __forceinline__ bool finite_val(float x) { return isfinite(x); }
// on the bits: a comparison would take the FP64 unit
__device__ __forceinline__ bool finite_val(double x) { return (__double2hiint(x) & 0x7FF00000) != 0x7FF00000; }

__device__ __forceinline__ uint32_t link_kind(uint32_t d) { return (d >> LINK_KIND_SHIFT) & 7u; }
__device__ __forceinline__ uint32_t link_row(uint32_t d) { return d >> LINK_ROW_SHIFT; }
__device__ __forceinline__ bool link_a_leaves(uint32_t d, int p) { return (d >> (LINK_PAIR_SHIFT + p)) & 1u; }
__device__ __forceinline__ bool link_boundary(uint32_t d) { return link_kind(d) - LK_WALL <= LK_SYMMETRY - LK_WALL; }
template <int MAXF> __device__ __forceinline__ uint32_t boundary_mask(const uint32_t* d) {
    uint32_t m = 0;
#pragma unroll
    for (int k = 0; k < MAXF; k++) m |= link_boundary(d[k]) ? 1u << k : 0u;
    return m;
}
// Boundary slots whose outgoing values are reconstructed (inlets, pressure
// outlets); on the others every face value is a ghost value (Sec. 2.4.2).
__device__ __forceinline__ bool kind_io(uint32_t kind) { return kind == LK_INLET || kind == LK_PRESSURE; }

template <typename T> __device__ __forceinline__ void to_pairs(const T* f, Pair<T>* p) {
#pragma unroll
    for (int q = 0; q < 4; q++) p[q] = make_pair2(f[dir_a(q)], f[dir_b(q)]);
}
template <typename T> __device__ __forceinline__ void from_pairs(const Pair<T>* p, T* f) {
#pragma unroll
    for (int q = 0; q < 4; q++) split2(p[q], f[dir_a(q)], f[dir_b(q)]);
}

// Slots (bit k) that some active thread of the warp uses: a polygon with
// fewer faces than MAXF leaves its last slots empty, and when every cell of a
// warp does (a warp of triangles in a 4-slot mesh), the warp skips them as a
// whole.  Slots 0..2 are always used.  Taken where the warp is whole: before any branch
// on what a cell is.
template <int MAXF>
__device__ __forceinline__ uint32_t warp_slots(const uint32_t* d) {
    uint32_t u = 7u;
#pragma unroll
    for (int k = 3; k < MAXF; k++)
        if (link_kind(d[k]) != LK_NONE) u |= 1u << k;
    return __reduce_or_sync(__activemask(), u);
}

// One slot's part of the least-squares gradient (Eq. leastsquare) of the eight
// moving directions: grad += c (f_neighbour - f), half h of the pairs (2 h, 2 h + 1).
template <typename T>
__device__ __forceinline__ void add_gradient(const Quad<T>& nb, const Pair<T>& cx, const Pair<T>& cy, int h,
                                             const Pair<T>* f, Pair<T>* gx, Pair<T>* gy) {
#pragma unroll
    for (int q = 0; q < 2; q++) {
        const int p = 2 * h + q;
        const Pair<T> dd = sub2(make_pair2(nb.v[2 * q], nb.v[2 * q + 1]), f[p]);
        gx[p] = fma2(cx, dd, gx[p]);
        gy[p] = fma2(cy, dd, gy[p]);
    }
}

// The values that leave a cell through one face (Eq. lslrflux): of each pair
// the direction that leaves, f + grad f . r.  FP32 computes both directions in
// one packed operation and picks; FP64, whose units are the limit (16 cycles
// per warp instruction and SM, whatever the active lanes), picks the operands
// first and computes four values instead of eight.
__device__ __forceinline__ Quad<float> leaving(uint32_t d, const Pair<float>* f, const Pair<float>* gx,
                                               const Pair<float>* gy, const float2& r) {
    const Pair<float> rx = make_pair2(r.x, r.x), ry = make_pair2(r.y, r.y);
    Quad<float> o;
#pragma unroll
    for (int p = 0; p < 4; p++) {
        float a, b;
        split2(fma2(gy[p], ry, fma2(gx[p], rx, f[p])), a, b);
        o.v[p] = link_a_leaves(d, p) ? a : b;
    }
    return o;
}
__device__ __forceinline__ Quad<double> leaving(uint32_t d, const Pair<double>* f, const Pair<double>* gx,
                                                const Pair<double>* gy, const double2& r) {
    Quad<double> o;
#pragma unroll
    for (int p = 0; p < 4; p++) {
        const bool s = link_a_leaves(d, p);
        o.v[p] = fma(s ? gy[p].x : gy[p].y, r.y, fma(s ? gx[p].x : gx[p].y, r.x, s ? f[p].x : f[p].y));
    }
    return o;
}

// One slot's part of the flux sum of Eq. (rhs): (e . n dl / A) times the face
// value of each direction (deviation mode: minus the cell's own value, the same
// in exact arithmetic because the face vectors of a closed cell sum to zero,
// without the rounding of the FP32 face vectors acting on the constant part of
// g).  out: what the cell sends through the face, in: what it receives.
template <typename T, bool DEV>
__device__ __forceinline__ void add_flux(uint32_t d, const typename Vec2<T>::type& n, const Quad<T>& out,
                                         const Quad<T>& in, const Pair<T>* f, Pair<T>* flux) {
    const T en[4] = {n.x, n.y, n.x + n.y, n.y - n.x};
#pragma unroll
    for (int p = 0; p < 4; p++) {
        const bool s = link_a_leaves(d, p);
        Pair<T> v = make_pair2(s ? out.v[p] : in.v[p], s ? in.v[p] : out.v[p]);
        if constexpr (DEV) v = sub2(v, f[p]);
        flux[p] = fma2(make_pair2(en[p], -en[p]), v, flux[p]);
    }
}

// Boundary slots of one cell (Sec. 2.4): the ghost differences enter the
// gradient; where the cell's faces are in the face table (own rows, and ghost
// rows for what enters), the boundary face values that are ghost values are
// written: everything on walls, symmetry planes (half way to the ghost) and
// external outlets, what enters on inlets and pressure outlets.  It needs the
// cell's own state only.
//   tag(k)  boundary tag, lsq(k) / face(k) vectors of slot k
//   own(k, q), in(k, link word, q)  store a row
// NEXT: each cell takes its next boundary slot, whichever that is, so that the
// cells of a warp that have one boundary face go through the code once, not once
// per slot number (the resident loop, where boundary warps are the critical
// path: 2.31 -> 2.00 us per stage of a 128^2 cavity).  The streaming kernels, where
// they are few and registers short, unroll the slots (NEXT costs 8% of a stage of the
// 256-instance batch: its slot number spills).
template <typename T, bool DEV, int MAXF, bool NEXT, typename Tag, typename Lsq, typename Face, typename Own, typename In>
__device__ __forceinline__ void boundary_slots(const uint32_t* d, const BcParam* bcs, T f0, const Pair<T>* fp,
                                               Pair<T>* gx, Pair<T>* gy, Tag tag, Lsq lsq, Face face, Own own, In in) {
    T f[FVLBM_Q];
    f[0] = f0;
    from_pairs(fp, f);
    T rho, ux, uy;
    moments<T, DEV>(f, rho, ux, uy);
    T fe[FVLBM_Q];
    if constexpr (!DEV) {   // once per cell: FP64 operations are dear, FP32 registers are
#pragma unroll
        for (int a = 1; a < FVLBM_Q; a++) fe[a] = feqs<T, DEV>(a, rho, ux, uy);
    }
    auto slot = [&](int k, uint32_t dk) {
        const Ghost<T> g = ghost_state<T, DEV>(link_kind(dk), bcs[tag(k)], rho, ux, uy, [&] { return face(k); });
        const typename Vec2<T>::type c = lsq(k);
        const Pair<T> cx = make_pair2(c.x, c.x), cy = make_pair2(c.y, c.y);
        const T part = g.sym ? T(0.5) : T(1);
        Quad<T> qo, qi;
#pragma unroll
        for (int p = 0; p < 4; p++) {
            const int a = dir_a(p), b = dir_b(p);
            const T da = ghost_delta<T, DEV>(g, a, f[a], DEV ? feqs<T, DEV>(a, rho, ux, uy) : fe[a]);
            const T db = ghost_delta<T, DEV>(g, b, f[b], DEV ? feqs<T, DEV>(b, rho, ux, uy) : fe[b]);
            const Pair<T> dd = make_pair2(da, db);
            gx[p] = fma2(cx, dd, gx[p]);
            gy[p] = fma2(cy, dd, gy[p]);
            // (a choice of factor spares FP64 an operation, a choice of result FP32 a register)
            const T va = !DEV ? fma(part, da, f[a]) : g.sym ? f[a] + T(0.5) * da : f[a] + da;
            const T vb = !DEV ? fma(part, db, f[b]) : g.sym ? f[b] + T(0.5) * db : f[b] + db;
            const bool s = link_a_leaves(dk, p);
            qo.v[p] = s ? va : vb;
            qi.v[p] = s ? vb : va;
        }
        in(k, dk, qi);
        if (!g.io) own(k, qo);
    };
    if constexpr (NEXT) {
        for (uint32_t left = boundary_mask<MAXF>(d); left; left &= left - 1) {
            const int k = __ffs(left) - 1;
            uint32_t dk = d[0];
#pragma unroll
            for (int q = 1; q < MAXF; q++) dk = k == q ? d[q] : dk;
            slot(k, dk);
        }
    } else {
#pragma unroll
        for (int k = 0; k < MAXF; k++)
            if (link_boundary(d[k])) slot(k, d[k]);
    }
}

// ------------------------------------------------------------------ FP64 by lanes
// Four lanes per cell, lane p with the pair p of its moving directions.  GB300
// has one FP64 unit per SM quarter, which takes 64 cycles for a warp's
// instruction whatever its active lanes (about 19 per SM when all four work):
// with a pair per lane a warp carries 8 cells through a quarter of the
// instructions, and its chain is a quarter as long.
__device__ __forceinline__ double lane_weight(int p) { return p < 2 ? 1.0 / 9.0 : 1.0 / 36.0; }
// rho, u of the four lanes' cell, in the order of moments() (every lane of the
// warp takes part)
__device__ __forceinline__ void lanes_moments(int p, double f0, double fa, double fb, double& rho, double& ux, double& uy) {
    const double S = fa + fb, Df = fa - fb;
    const double s1 = S + __shfl_xor_sync(0xFFFFFFFFu, S, 1);
    rho = f0 + (s1 + __shfl_xor_sync(0xFFFFFFFFu, s1, 2));
    const double o = __shfl_xor_sync(0xFFFFFFFFu, Df, 1);
    const double even = (p & 1) ? o : Df, odd = (p & 1) ? Df : o;
    const double X = p >= 2 ? even - odd : even, Y = p >= 2 ? even + odd : odd;
    const double mx = X + __shfl_xor_sync(0xFFFFFFFFu, X, 2), my = Y + __shfl_xor_sync(0xFFFFFFFFu, Y, 2);
    const double inv_rho = 1.0 / rho;
    ux = mul_rn(mx, inv_rho);
    uy = mul_rn(my, inv_rho);
}
// f^eq / (rho w) of the lane's two directions and of direction 0
__device__ __forceinline__ void lane_eq(int p, double ux, double uy, double& qa, double& qb, double& q0) {
    const double diag = uy + (p == 3 ? -ux : ux);
    const double eu = p == 0 ? ux : p == 1 ? uy : diag;
    q0 = fma(-1.5, square(ux, uy), 1.0);
    qa = fma(eu, fma(4.5, eu, 3.0), q0);
    qb = fma(eu, fma(4.5, eu, -3.0), q0);
}
// boundary_slots() for the lane's pair; qa, qb: lane_eq of the cell.
template <int MAXF, typename Tag, typename Lsq, typename Face, typename Own, typename In>
__device__ __forceinline__ void lane_boundary(int p, const uint32_t* d, const BcParam* bcs, double fa, double fb, double rho,
                                              double ux, double uy, double qa, double qb, double& gax, double& gay,
                                              double& gbx, double& gby, Tag tag, Lsq lsq, Face face, Own own, In in) {
    const double w = lane_weight(p), rw = rho * w, ea = mul_rn(rw, qa), eb = mul_rn(rw, qb);
    for (uint32_t left = boundary_mask<MAXF>(d); left; left &= left - 1) {
        const int k = __ffs(left) - 1;
        uint32_t dk = d[0];
#pragma unroll
        for (int z = 1; z < MAXF; z++) dk = k == z ? d[z] : dk;
        const double2 c = lsq(k);
        const Ghost<double> g = ghost_state<double, false>(link_kind(dk), bcs[tag(k)], rho, ux, uy, [&] { return face(k); });
        double ga, gb, g0, da = 0, db = 0;
        if (!g.zero) {
            lane_eq(p, g.ux, g.uy, ga, gb, g0);
            const double gw = g.r * w;
            da = fma(gw, ga, g.sym ? -fa : -ea);
            db = fma(gw, gb, g.sym ? -fb : -eb);
        }
        gax = fma(c.x, da, gax);
        gay = fma(c.y, da, gay);
        gbx = fma(c.x, db, gbx);
        gby = fma(c.y, db, gby);
        const double part = g.sym ? 0.5 : 1.0, va = fma(part, da, fa), vb = fma(part, db, fb);
        const bool a_leaves = link_a_leaves(dk, p);
        in(k, dk, a_leaves ? vb : va);
        if (!g.io) own(k, a_leaves ? va : vb);
    }
}

// cp.async copy of one 16- or 8-byte element from global to shared memory
// (16 bytes: past L1).
template <int BYTES>
__device__ __forceinline__ void cp_async_elem(void* dst, const void* src) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(src) : "memory");
}
// Hint: bring a 16-byte aligned range (a multiple of 16 bytes) into L2.
__device__ __forceinline__ void prefetch_l2(const void* p, int64_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(p), "r"((uint32_t)bytes) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
// Collision and time update of one cell (Eq. rhs, Sec. 2.3): rhs = -flux -
// (f - f^eq) / tau, in two parts.  The first needs the cell's own state only:
//   FP64: col = f^eq - f, f^eq_a = rho w_a q_a, q_a = e.u (4.5 e.u + 3) + 1 - 1.5 u^2;
//         the units that do this are the limit, so no operation is spent that a
//         fused multiply-add can absorb
//   deviation modes: col = f - f^eq (the sign that makes every packed operation
//         one fused multiply-add).  It carries no mass or momentum (f^eq has the
//         cell's rho and rho u), so directions 0..2 follow from directions 3..8
//         through those identities.  Evaluated directly in FP32, its nine rounding
//         errors (about eps |g| each, |g| >> |f^eq - f|) would add a spurious mass
//         and momentum source of about eps |g| / tau per unit time, which
//         dominated the velocity error at small tau.
template <typename T, bool DEV>
__device__ __forceinline__ void collision(const T* f, T* col) {
    T rho, ux, uy;
    moments<T, DEV>(f, rho, ux, uy);
    const T eu[4] = {ux, uy, ux + uy, uy - ux};   // e_A . u of the pairs
    if constexpr (!DEV) {
        const T q0 = fma(T(-1.5), square(ux, uy), T(1));
        const T rw[3] = {rho * T(4.0 / 9.0), rho * T(1.0 / 9.0), rho * T(1.0 / 36.0)};
        col[0] = fma(rw[0], q0, -f[0]);
#pragma unroll
        for (int p = 0; p < 4; p++) {
            const int a = dir_a(p), b = dir_b(p);
            col[a] = fma(rw[p < 2 ? 1 : 2], fma(eu[p], fma(T(4.5), eu[p], T(3)), q0), -f[a]);
            col[b] = fma(rw[p < 2 ? 1 : 2], fma(eu[p], fma(T(4.5), eu[p], T(-3)), q0), -f[b]);
        }
    } else {
        const T uu15 = T(1.5) * square(ux, uy);
        const Pair<T> r2 = make_pair2(rho, rho), r1 = make_pair2(T(1) + rho, T(1) + rho);
        const Pair<T> c45 = make_pair2(T(4.5), T(4.5)), c3 = make_pair2(T(3), T(3)), cu = make_pair2(-uu15, -uu15);
#pragma unroll
        for (int p = 2; p < 4; p++) {
            const Pair<T> e = make_pair2(eu[p], -eu[p]);
            const Pair<T> q = fma2(r1, fma2(e, fma2(c45, e, c3), cu), r2);
            split2(fma2(make_pair2(T(-1.0 / 36.0), T(-1.0 / 36.0)), q, make_pair2(f[dir_a(p)], f[dir_b(p)])),
                   col[dir_a(p)], col[dir_b(p)]);
        }
        {   // directions 3 and 4
            const Pair<T> e = make_pair2(-ux, -uy);
            const Pair<T> q = fma2(r1, fma2(e, fma2(c45, e, c3), cu), r2);
            split2(fma2(make_pair2(T(-1.0 / 9.0), T(-1.0 / 9.0)), q, make_pair2(f[3], f[4])), col[3], col[4]);
        }
        col[1] = col[3] - col[5] + col[6] + col[7] - col[8];
        col[2] = col[4] - col[5] - col[6] + col[7] + col[8];
        col[0] = -(col[1] + col[2] + col[3] + col[4] + col[5] + col[6] + col[7] + col[8]);
    }
}

// The second part: out = base + beta dt rhs (multistage) or the AB2
// combination with rp, the previous right-hand side (replaced by this one).
// Returns false when an output is not finite.
template <typename T> struct Relax {
    T inv_tau, dt;
    __device__ __forceinline__ explicit Relax(const InstParam& P) : inv_tau(inst_inv_tau<T>(P)), dt(inst_dt<T>(P)) {}
};
template <typename T, bool DEV>
__device__ __forceinline__ bool advance(const Relax<T>& P, const T* f, const T* col, const Pair<T>* flux,
                                        const T* base, T* rp, T beta, int mode, T* out) {
    const T inv_tau = P.inv_tau, dt = P.dt;
    T fl[FVLBM_Q];
    fl[0] = T(0);
    from_pairs(flux, fl);
    if (mode == MODE_RK) {
        const T c1 = beta * dt;
        if constexpr (!DEV) {
            const T c2 = c1 * inv_tau;   // base + c1 (-flux + col / tau)
#pragma unroll
            for (int a = 0; a < FVLBM_Q; a++) out[a] = fma(c2, col[a], a == 0 ? base[a] : fma(-c1, fl[a], base[a]));
        } else {
            const Pair<T> it = make_pair2(inv_tau, inv_tau), c = make_pair2(-c1, -c1);
            out[0] = fma(-c1, mul_rn(col[0], inv_tau), base[0]);
#pragma unroll
            for (int p = 0; p < 4; p++)
                split2(fma2(c, fma2(make_pair2(col[dir_a(p)], col[dir_b(p)]), it, flux[p]),
                            make_pair2(base[dir_a(p)], base[dir_b(p)])), out[dir_a(p)], out[dir_b(p)]);
        }
    } else {
#pragma unroll
        for (int a = 0; a < FVLBM_Q; a++) {
            const T rhs = DEV ? -fma(col[a], inv_tau, fl[a]) : fma(inv_tau, col[a], -fl[a]);
            out[a] = fma(dt, mode == MODE_AB2_FIRST ? rhs : fma(T(1.5), rhs, T(-0.5) * rp[a]), f[a]);
            rp[a] = rhs;
        }
    }
    if constexpr (!DEV) {   // tests on the bits: the FP64 units have enough to do
        bool ok = true;
#pragma unroll
        for (int a = 0; a < FVLBM_Q; a++) ok &= finite_val(out[a]);
        return ok;
    }
    // one test: the sum of the outputs is not finite when any output is not
    T sum = out[0];
#pragma unroll
    for (int a = 1; a < FVLBM_Q; a++) sum += out[a];
    return finite_val(sum);
}

// The history of cell i (AB2).
template <typename T, typename I> __device__ __forceinline__ void load_history(const DevView& v, I i, T* rp) {
#pragma unroll
    for (int a = 0; a < FVLBM_Q; a++) rp[a] = ((const T*)v.rprev)[a * v.np + i];
}
template <typename T, typename I> __device__ __forceinline__ void store_history(const DevView& v, I i, const T* rp) {
#pragma unroll
    for (int a = 0; a < FVLBM_Q; a++) ((T*)v.rprev)[a * v.np + i] = rp[a];
}

// ------------------------------------------------------------------ kernels
// Two-kernel stage (default in FP64, where the FP64 units bound it: 2.77 ms per
// stage of the 6.67 M cell batch; 4.10 with eight reconstructed values per face,
// products with zero velocity components and finiteness compared in FP64).  The
// face table holds, for every (cell, slot), the four
// values that leave the cell there (one side of each (face, direction) is its
// only writer, with no test of who writes: a warp stores whole rows), then
// the ghost records.  Row of (cell i, slot k): blk_index(i, MAXF) + k * BLK.
template <typename T> __device__ __forceinline__ typename Vec16<T>::type* face_row(void* fv, int64_t row) {
    return (typename Vec16<T>::type*)fv + row * QUAD_UNITS<T>;
}

// Kernel 1 (Steps 1-3): per cell the gradient, then what leaves it through
// every face, and the ghost values of its boundary faces.
template <typename T, typename S, int MAXF, bool DEV>
__global__ void __launch_bounds__(256) face_values_kernel(DevView v, const S* __restrict__ fin) {
    typedef typename Vec2<T>::type T2;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= v.n_grad) return;   // owned cells and, in a partition, the first ghost ring
    const GeoRef<T, MAXF> G(v.geo, i);
    uint32_t d[MAXF];
    load_links<MAXF>(v.link, i, d);
    int32_t nb[MAXF];
    load_links<MAXF>((const uint4*)v.nbr, i, (uint32_t*)nb);
    T f[FVLBM_Q];
    CellIO<S>::template load<T, DEV>(fin, i, v.inst[v.grp[i]], f);
    Pair<T> fp[4], gx[4], gy[4];
    to_pairs(f, fp);
#pragma unroll
    for (int p = 0; p < 4; p++) gx[p] = gy[p] = make_pair2(T(0), T(0));
    const uint32_t used = warp_slots<MAXF>(d);
    const int64_t row = blk_index(i, MAXF);
    auto boundary = [&] {
        if (boundary_mask<MAXF>(d))
            boundary_slots<T, DEV, MAXF, false>(d, v.bc, f[0], fp, gx, gy, [&](int k) { return v.bctag[i * MAXF + k]; },
                                         [&](int k) { return G.get(GEO_LSQ, k); }, [&](int k) { return G.get(GEO_FACE, k); },
                                         [&](int k, const Quad<T>& q) { store_quad(face_row<T>(v.fv, row + k * BLK), 1, q); },
                                         [&](int k, uint32_t, const Quad<T>& q) {
                                             if (i < v.n_cell) store_quad(face_row<T>(v.fv, v.np * MAXF + nb[k]), 1, q);
                                         });
    };
    if (!DEV) boundary();
#pragma unroll
    for (int k = 0; k < MAXF; k++) {
        if (k >= 3 && !((used >> k) & 1u)) continue;
        const int64_t j = link_boundary(d[k]) ? i : (int64_t)nb[k];
        T fj[FVLBM_Q];
        CellIO<S>::template load<T, DEV>(fin, j, v.inst[v.grp[j]], fj);
        const T2 c = G.get(GEO_LSQ, k);
        const Pair<T> cx = make_pair2(c.x, c.x), cy = make_pair2(c.y, c.y);
#pragma unroll
        for (int h = 0; h < 2; h++)
            add_gradient(Quad<T>{{fj[dir_a(2 * h)], fj[dir_b(2 * h)], fj[dir_a(2 * h + 1)], fj[dir_b(2 * h + 1)]}}, cx,
                         cy, h, fp, gx, gy);
    }
    if (DEV) boundary();
#pragma unroll
    for (int k = 0; k < MAXF; k++) {
        if (k >= 3 && !((used >> k) & 1u)) continue;
        const uint32_t kind = link_kind(d[k]);
        if (kind >= LK_WALL && !kind_io(kind)) continue;   // ghost values, or no face
        store_quad(face_row<T>(v.fv, row + k * BLK), 1, leaving(d[k], fp, gx, gy, G.get(GEO_MID, k)));
    }
}

// Kernel 1 in FP64, four lanes per cell: the same values.
template <int MAXF>
__global__ void __launch_bounds__(256) face_values_pairs_kernel(DevView v, const double* __restrict__ fin) {
    const int p = threadIdx.x & 3;
    const int64_t at = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
    const bool ours = at < v.n_grad;   // owned cells and, in a partition, the first ghost ring
    const int64_t i = ours ? at : v.n_grad - 1;
    const GeoRef<double, MAXF> G(v.geo, i);
    uint32_t d[MAXF];
    load_links<MAXF>(v.link, i, d);
    int32_t nb[MAXF];
    load_links<MAXF>((const uint4*)v.nbr, i, (uint32_t*)nb);
    const double2 f = CellIO<double>::pairs(fin, i)[p * BLK];
    const int64_t row = blk_index(i, MAXF);
    double* fv = (double*)v.fv + p;
    double gax = 0, gay = 0, gbx = 0, gby = 0;
    const bool edge = boundary_mask<MAXF>(d) != 0;
    const uint32_t used = warp_slots<MAXF>(d);
    if (__any_sync(0xFFFFFFFFu, edge)) {
        double rho, ux, uy, qa, qb, q0;
        lanes_moments(p, *CellIO<double>::rest(fin, i), f.x, f.y, rho, ux, uy);
        lane_eq(p, ux, uy, qa, qb, q0);
        if (edge)
            lane_boundary<MAXF>(p, d, v.bc, f.x, f.y, rho, ux, uy, qa, qb, gax, gay, gbx, gby,
                                [&](int k) { return v.bctag[i * MAXF + k]; }, [&](int k) { return G.get(GEO_LSQ, k); },
                                [&](int k) { return G.get(GEO_FACE, k); },
                                [&](int k, double z) { if (ours) fv[(row + k * BLK) * 4] = z; },
                                [&](int k, uint32_t, double z) {
                                    if (!ours || i >= v.n_cell) return;
                                    int32_t ghost = nb[0];
#pragma unroll
                                    for (int x = 1; x < MAXF; x++) ghost = k == x ? nb[x] : ghost;
                                    fv[(v.np * MAXF + ghost) * 4] = z;
                                });
    }
#pragma unroll
    for (int k = 0; k < MAXF; k++) {
        if (k >= 3 && !((used >> k) & 1u)) continue;
        const double2 n = CellIO<double>::pairs(fin, link_boundary(d[k]) ? i : (int64_t)nb[k])[p * BLK];
        const double2 c = G.get(GEO_LSQ, k);
        const double da = n.x - f.x, db = n.y - f.y;
        gax = fma(c.x, da, gax);
        gay = fma(c.y, da, gay);
        gbx = fma(c.x, db, gbx);
        gby = fma(c.y, db, gby);
    }
#pragma unroll
    for (int k = 0; k < MAXF; k++) {
        if (k >= 3 && !((used >> k) & 1u)) continue;
        const uint32_t kind = link_kind(d[k]);
        if (kind >= LK_WALL && !kind_io(kind)) continue;   // ghost values, or no face
        const double2 m = G.get(GEO_MID, k);
        const bool a = link_a_leaves(d[k], p);
        const double z = fma(a ? gay : gby, m.y, fma(a ? gax : gbx, m.x, a ? f.x : f.y));
        if (ours) fv[(row + k * BLK) * 4] = z;
    }
}

// Kernel 2 (Steps 4-5): flux sum over the cell's faces, collision and time
// update.
template <typename T, typename S, int MAXF, bool DEV>
__global__ void __launch_bounds__(256) update_kernel(DevView v, const S* __restrict__ fin, const S* fbase, S* fout,
                                                     T beta, int mode) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= v.n_cell) return;
    const InstParam& P = v.inst[v.grp[i]];
    const GeoRef<T, MAXF> G(v.geo, i);
    uint32_t d[MAXF];
    load_links<MAXF>(v.link, i, d);
    int32_t nb[MAXF];
    load_links<MAXF>((const uint4*)v.nbr, i, (uint32_t*)nb);
    T f[FVLBM_Q];
    CellIO<S>::template load<T, DEV>(fin, i, P, f);
    Pair<T> fp[4], fx[4];
    to_pairs(f, fp);
#pragma unroll
    for (int p = 0; p < 4; p++) fx[p] = make_pair2(T(0), T(0));
    const int64_t row = blk_index(i, MAXF);
#pragma unroll
    for (int k = 0; k < MAXF; k++) {
        if (link_kind(d[k]) == LK_NONE) continue;
        const int64_t from = link_boundary(d[k]) ? v.np * MAXF + nb[k]
                                                 : blk_index((int64_t)nb[k], MAXF) + (int64_t)link_row(d[k]) * BLK;
        add_flux<T, DEV>(d[k], G.get(GEO_FACE, k), load_quad(face_row<T>(v.fv, row + k * BLK), 1),
                         load_quad(face_row<T>(v.fv, from), 1), fp, fx);
    }
    T fb[FVLBM_Q], rp[FVLBM_Q], col[FVLBM_Q], out[FVLBM_Q];
    const bool rk_base = mode == MODE_RK && fbase != fin;
    if (rk_base) CellIO<S>::template load<T, DEV>(fbase, i, P, fb);
    if (mode == MODE_AB2) load_history(v, i, rp);
    collision<T, DEV>(f, col);
    if (!advance<T, DEV>(Relax<T>(P), f, col, fx, rk_base ? fb : f, rp, beta, mode, out)) *v.flag = 1;
    if (mode != MODE_RK) store_history(v, i, rp);
    CellIO<S>::template store<T, DEV>(fout, i, P, out);
}

// Phase 2 of a tile for local cell l.  Boundary cells' part: ghost differences
// into the gradient and ghost values into the face table (rows that only the
// cell itself reads).
template <typename T, bool DEV, int MAXF, int TILE, bool NEXT, typename Lsq, typename Face>
__device__ __forceinline__ void tile_boundary(const BcParam* bc, const uint16_t* bctag, const uint32_t* d, uint32_t gl, T f0,
                                              const Pair<T>* f, Pair<T>* gx, Pair<T>* gy, typename Vec16<T>::type* tab,
                                              int l, bool mine, Lsq lsq, Face face) {
    constexpr int ROWS = TileDims<TILE, MAXF, sizeof(T)>::ROWS;
    boundary_slots<T, DEV, MAXF, NEXT>(d, bc, f0, f, gx, gy, [&](int k) { return bctag[(int64_t)gl * MAXF + k]; }, lsq, face,
                                       [&](int k, const Quad<T>& q) { store_quad(tab + k * TILE + l, ROWS, q); },
                                       [&](int, uint32_t dk, const Quad<T>& q) {
                                           if (mine) store_quad(tab + link_row(dk), ROWS, q);
                                       });
}
// All of it: the neighbour differences, boundary() where it adds its part, then
// what leaves the cell through every face into the face table.  lsq, mid: its
// geometry vectors by slot (mid after before_mid()).
template <typename T, bool DEV, int MAXF, int TILE, typename Lsq, typename Mid, typename BeforeMid, typename Boundary>
__device__ __forceinline__ void tile_faces(const uint32_t* d, const Pair<T>* f, Pair<T>* gx, Pair<T>* gy,
                                           const typename Vec16<T>::type* fs, typename Vec16<T>::type* tab, int l, Lsq lsq,
                                           Mid mid, BeforeMid before_mid, Boundary boundary) {
    typedef TileDims<TILE, MAXF, sizeof(T)> D;
    typedef typename Vec2<T>::type T2;
    constexpr int LS = D::LS, ROWS = D::ROWS, SU = 8 / Vec16<T>::N;
    // (FP64: before the neighbours, as the four-lane kernels, where it overlaps the wait for the halo)
#pragma unroll
    for (int p = 0; p < 4; p++) gx[p] = gy[p] = make_pair2(T(0), T(0));
    const bool bc = boundary_mask<MAXF>(d) != 0;
    // before the branch: every row that phase 3 reads for a warp has to be written here,
    // an empty slot's among them, also should the warp not come together after it
    const uint32_t used = warp_slots<MAXF>(d);
    if (!DEV && bc) boundary();
#pragma unroll
    for (int k = 0; k < MAXF; k++) {
        if (k >= 3 && !((used >> k) & 1u)) continue;
        const T2 ck = lsq(k);
        const Pair<T> cx = make_pair2(ck.x, ck.x), cy = make_pair2(ck.y, ck.y);
        const typename Vec16<T>::type* nb = fs + (d[k] & LINK_NB_MASK);
#pragma unroll
        for (int h = 0; h < 2; h++) add_gradient(load_quad(nb + h * (SU / 2) * LS, LS), cx, cy, h, f, gx, gy);
    }
    if (DEV && bc) boundary();
    before_mid();
#pragma unroll
    for (int k = 0; k < MAXF; k++) {
        if (k >= 3 && !((used >> k) & 1u)) continue;
        // ghost values are in place, a 1-ring cell's other faces are not the tile's;
        // an unused slot among used ones writes its (finite) state, read with weight zero
        const uint32_t kind = link_kind(d[k]);
        if (kind == LK_FLOW || kind == LK_NONE || kind_io(kind))
            store_quad(tab + k * TILE + l, ROWS, leaving(d[k], f, gx, gy, mid(k)));
    }
}

// Fused stage: one CTA per tile of consecutive cells (Hilbert order; tile
// and 1-ring together at most TILE cells), everything between the state read
// and the state write in shared memory:
//   phase 1  the moving directions of the tile, its 1-ring and its 2-ring into
//            shared memory (16-byte cp.async; the 16-bit formats raw, each cell
//            decoded by the thread that staged it); links and least-squares
//            vectors of each thread's gradient cell into registers
//   phase 2  per tile and 1-ring cell (one per thread): the gradient
//            (Eq. leastsquare) and, per face, the four values that leave the
//            cell there (Eq. lslrflux), as one 16-byte row of the face table (row
//            k * TILE + x: no bank conflict); boundary cells also their ghost
//            values (Sec. 2.4.2).  A tile cell's thread keeps its state
//   phase 3  per tile cell: per face its own row and the neighbour's (or
//            ghost) row give all eight face values; flux sum, collision and
//            the time update (Eq. rhs, Sec. 2.3)
// The global loads of each phase are issued before the barrier that precedes
// it, so that their latency overlaps the wait, and each CTA prefetches into L2
// the data of a tile that starts somewhat under one CTA lifetime later (pf =
// 5/8 of the resident CTAs ahead).  Shared-memory strides are compile-time
// constants (TileDims); the planner keeps every tile within them.
// Bound by latency (record -> halo list -> state, the two barriers) at the 32
// warps per SM that 64 registers allow, not by DRAM or issue: 256-instance
// batch (6.67 M cells) 0.281 ms per FP32 stage and 0.339 per FP16 stage (graph
// replay); with single 4-byte accesses, a table of faces and scalar arithmetic, half
// as many instructions again, 0.302 and 0.364.
constexpr int stage_ctas(int tile, int rsize) { return tile <= (rsize == 4 ? 1024 : 512) ? (rsize == 4 ? 1024 : 512) / tile : 1; }

template <typename T, typename S, int MAXF, bool DEV, int TILE>
__global__ void __launch_bounds__(TILE, stage_ctas(TILE, sizeof(T)))
    stage_tile_kernel(DevView v, const S* __restrict__ fin, const S* fbase, S* fout, T beta, int mode, int pf) {
    typedef TileDims<TILE, MAXF, sizeof(T)> D;
    typedef typename Vec2<T>::type T2;
    typedef typename Vec16<T>::type V;
    constexpr int LS = D::LS, ROWS = D::ROWS;
    constexpr int SU = 8 / Vec16<T>::N;      // 16-byte units of a cell's moving directions
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* fs = (V*)smem_raw;         // [SU][LS]         moving directions of the local cells
    V* tab = fs + SU * LS;        // [QUAD_UNITS][ROWS]  face table
    // cell, halo and 1-ring indices in 32 bits: the set-up keeps every array
    // of a fused-stage solver below 2^32 elements
    const uint32_t t = blockIdx.x;
    const int4 ra = ((const int4*)(v.tiles + t))[0], rb = ((const int4*)(v.tiles + t))[1];
    const uint32_t c0 = ra.x, h0 = ra.z, q0 = rb.x;
    const int nt = ra.y, nh = ra.w, n1 = rb.y, inst = rb.z;
    const int l = threadIdx.x;
    const bool mine = l < nt;          // this thread owns tile cell l
    const uint32_t gi = c0 + l;

    // phase 1 (thread l's first local cell is local cell l).  The 16-bit split
    // formats are staged raw in the face-table area, which is free until phase 2.
    constexpr bool PLAIN = sizeof(S) == sizeof(T);
    uint4* rawh = (uint4*)tab;                     // [LS]
    uint2* rawt = (uint2*)(rawh + LS);             // [LS]
    static_assert(PLAIN || LS * 24 <= ROWS * 4 * (int)sizeof(T), "raw staging fits the face table");
    const int n2 = nt + n1;            // gradient cells: the planner keeps nt + n1 <= TILE
    // a thread stages at most two local cells (LS <= 2 TILE)
    static_assert(LS <= 2 * TILE, "two local cells per thread");
    const int n_local = nt + nh;
    uint32_t gl = c0, gl2 = 0;
    if (l < n_local) gl = mine ? gi : (uint32_t)v.halo[h0 + (l - nt)];
    if (l + TILE < n_local) gl2 = (uint32_t)v.halo[h0 + (l + TILE - nt)];
    // phase 2 gives local cell x (tile cell, or 1-ring entry x - nt) to thread x
    uint32_t d[MAXF];
    T2 c[MAXF];
    const GeoRef<T, MAXF> G(v.geo, gl);
    if (l < n2) {
        if (mine) {
            load_links<MAXF>(v.link, gi, d);
        } else {
#pragma unroll
            for (int u = 0; u < MAXF / 4; u++) {
                const uint4 x = v.r1link[u * v.n_r1 + q0 + (l - nt)];
                d[4 * u] = x.x;
                d[4 * u + 1] = x.y;
                d[4 * u + 2] = x.z;
                d[4 * u + 3] = x.w;
            }
        }
        if constexpr (MAXF <= 4) G.load(GEO_LSQ, c);
    }
    T f0 = T(0);
    auto stage_cell = [&](int x, uint32_t gx) {
        if constexpr (PLAIN) {
            const V* p = (const V*)CellIO<S>::pairs(fin, gx);
#pragma unroll
            for (int u = 0; u < SU; u++) cp_async_elem<16>(fs + u * LS + x, p + u * BLK);
        } else {
            cp_async_elem<16>(rawh + x, CellIO<S>::head(fin, gx));
            cp_async_elem<8>(rawt + x, CellIO<S>::tail(fin, gx));
        }
    };
    if (l < n_local) stage_cell(l, gl);
    if (l + TILE < n_local) stage_cell(l + TILE, gl2);
    if constexpr (PLAIN)
        if (l < n2) f0 = (T)*CellIO<S>::rest(fin, gl);
    // A CTA that starts somewhat before this one ends works on about tile
    // t + pf (pf = 5/8 of the CTAs resident on the GPU): bring that tile's
    // state and geometry into L2 now, so that its staging reads L2 rather than
    // HBM.  The last thread does it once its own copies are in flight, so that
    // the loads of the other tile's bounds overlap them.
    if (l == TILE - 1 && pf > 0 && t + pf < v.n_tiles) {
        const TileRec R = v.tiles[t + pf];
        const int64_t b0 = R.c0 >> BLK_SHIFT;
        const int64_t nb = ((R.c0 + R.nt + BLK - 1) >> BLK_SHIFT) - b0;
        constexpr int64_t SB = CellIO<S>::BLOCK_BYTES;
        constexpr int64_t DB = (int64_t)MAXF * BLK * sizeof(uint32_t);
        constexpr int64_t GB = (int64_t)3 * MAXF * BLK * sizeof(T2);
        prefetch_l2((const unsigned char*)fin + b0 * SB, nb * SB);
        if (mode == MODE_RK && fbase != fin) prefetch_l2((const unsigned char*)fbase + b0 * SB, nb * SB);
        prefetch_l2((const unsigned char*)v.link + b0 * DB, nb * DB);
        prefetch_l2((const unsigned char*)v.geo + b0 * GB, nb * GB);
        // its halo list and 1-ring links (16-byte aligned cover of each range)
        auto range = [&](const void* base, int64_t begin, int64_t end) {
            const int64_t a = begin & ~(int64_t)15, e = (end + 15) & ~(int64_t)15;
            if (e > a) prefetch_l2((const unsigned char*)base + a, e - a);
        };
        range(v.halo, 4 * (int64_t)R.h0, 4 * (int64_t)(R.h0 + R.nh));
#pragma unroll
        for (int u = 0; u < MAXF / 4; u++)
            range(v.r1link + u * v.n_r1, 16 * (int64_t)R.q0, 16 * (int64_t)(R.q0 + R.n1));
        if (R.inst < 0) range(v.grp, 4 * (int64_t)R.c0, 4 * (int64_t)(R.c0 + R.nt));
    }
    cp_async_wait_all();
    // a 16-bit state is decoded by the thread that staged it (its own copies
    // are complete after the wait), so one barrier serves both
    if constexpr (!PLAIN) {
        auto decode_cell = [&](int x, uint32_t gx, T& rest) {
            T f[FVLBM_Q];
            CellIO<S>::template decode<T>(rawh[x], rawt[x], v.inst[inst >= 0 ? inst : v.grp[gx]], f);
            rest = f[0];
#pragma unroll
            for (int h = 0; h < 2; h++)
                store_quad(fs + h * (SU / 2) * LS + x, LS,
                           Quad<T>{{f[dir_a(2 * h)], f[dir_b(2 * h)], f[dir_a(2 * h + 1)], f[dir_b(2 * h + 1)]}});
        };
        T none;
        if (l < n_local) decode_cell(l, gl, f0);
        if (l + TILE < n_local) decode_cell(l + TILE, gl2, none);
    }
    __syncthreads();

    // phase 2 (a tile cell's thread keeps its state for phase 3)
    Pair<T> f[4];
    if (l < n2) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const Quad<T> q = load_quad(fs + h * (SU / 2) * LS + l, LS);
            f[2 * h] = make_pair2(q.v[0], q.v[1]);
            f[2 * h + 1] = make_pair2(q.v[2], q.v[3]);
        }
        auto lsq = [&](int k) { return MAXF <= 4 ? c[k] : G.get(GEO_LSQ, k); };
        Pair<T> gx[4], gy[4];
        tile_faces<T, DEV, MAXF, TILE>(d, f, gx, gy, fs, tab, l, lsq, [&](int k) { return G.get(GEO_MID, k); }, [] {}, [&] {
            tile_boundary<T, DEV, MAXF, TILE, false>(v.bc, v.bctag, d, gl, f0, f, gx, gy, tab, l, mine, lsq,
                                                     [&](int k) { return G.get(GEO_FACE, k); });
        });
    }
    // phase 3 inputs, in flight during the wait
    T2 n[MAXF];
    T fb[FVLBM_Q];
    const bool rk_base = mode == MODE_RK && fbase != fin;
    if (mine) {
        G.load(GEO_FACE, n);
        if (rk_base) CellIO<S>::template load<T, DEV>(fbase, gi, v.inst[inst >= 0 ? inst : v.grp[gi]], fb);
    }
    __syncthreads();

    if (!mine) return;
    const InstParam& P = v.inst[inst >= 0 ? inst : v.grp[gi]];
    Pair<T> fx[4];
#pragma unroll
    for (int p = 0; p < 4; p++) fx[p] = make_pair2(T(0), T(0));
    const uint32_t used = warp_slots<MAXF>(d);
#pragma unroll
    for (int k = 0; k < MAXF; k++) {
        if (k >= 3 && !((used >> k) & 1u)) continue;
        add_flux<T, DEV>(d[k], n[k], load_quad(tab + k * TILE + l, ROWS), load_quad(tab + link_row(d[k]), ROWS), f, fx);
    }
    T fa[FVLBM_Q], rp[FVLBM_Q], col[FVLBM_Q], out[FVLBM_Q];
    fa[0] = f0;
    from_pairs(f, fa);
    if (!rk_base) {
#pragma unroll
        for (int a = 0; a < FVLBM_Q; a++) fb[a] = fa[a];
    }
    if (mode == MODE_AB2) load_history(v, gi, rp);
    collision<T, DEV>(fa, col);
    if (!advance<T, DEV>(Relax<T>(P), fa, col, fx, fb, rp, beta, mode, out)) *v.flag = 1;
    if (mode != MODE_RK) store_history(v, gi, rp);
    CellIO<S>::template store<T, DEV>(fout, gi, P, out);
}

static inline unsigned grid_of(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

static inline int check_launch(const char* what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(FVLBM_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
    return FVLBM_OK;
}

template <typename T, typename S, int MAXF, bool DEV, int TILE>
static int tile_launch(const DevView& v, cudaStream_t st, const void* fin, const void* fbase, void* fout,
                       double beta, int mode) {
    auto kern = stage_tile_kernel<T, S, MAXF, DEV, TILE>;
    typedef TileDims<TILE, MAXF, sizeof(T)> D;
    constexpr size_t base = D::BYTES, most = D::MAX_BYTES;
    const size_t smem = base + (v.tile_ghosts > D::GHOSTS ? (size_t)4 * sizeof(T) * (v.tile_ghosts - D::GHOSTS) : 0);
    if (most > 48 * 1024) {   // the most of any plan: solvers of several threads share the attribute
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
        if (e != cudaSuccess) return fail(FVLBM_ERR_CUDA, "fused stage: %zu B shared memory: %s", most, cudaGetErrorString(e));
    }
    // prefetch distance: 5/8 of the CTAs that fit on the GPU at once (queried
    // once per kernel; a function-local static is initialised once even when
    // several host threads launch at the same time).  Measured on GB300 over
    // 0.5 to 1.5 times the resident CTAs: 0.6 to 0.75 was best, longer
    // distances let the prefetched lines age out of L2 before their tile runs.
    static const int per_sm = [&] {
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, TILE, base) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        return n;
    }();
    const int pf = per_sm * v.sms * 5 / 8;
    kern<<<(unsigned)v.n_tiles, TILE, smem, st>>>(v, (const S*)fin, (const S*)fbase, (S*)fout, (T)beta, mode, pf);
    return FVLBM_OK;
}

// Tile sizes whose shared memory exceeds a CTA's are not instantiated (the
// planner never selects them).
constexpr size_t TILE_SMEM_LIMIT = 227 * 1024;

template <typename T, typename S, int MAXF, bool DEV, int TILE>
static int tile_launch_if_fits(const DevView& v, cudaStream_t st, const void* fin, const void* fbase, void* fout,
                               double beta, int mode) {
    static_assert(sizeof(T) == 8 || TileDims<TILE, MAXF, sizeof(T)>::MAX_BYTES <= TILE_SMEM_LIMIT, "every plan fits");
    if constexpr (TileDims<TILE, MAXF, sizeof(T)>::BYTES <= TILE_SMEM_LIMIT)
        return tile_launch<T, S, MAXF, DEV, TILE>(v, st, fin, fbase, fout, beta, mode);
    return fail(FVLBM_ERR_UNSUPPORTED, "tile size %d does not fit in shared memory", TILE);
}

template <typename T, typename S, int MAXF, bool DEV>
static int tile_dispatch(const DevView& v, cudaStream_t st, const void* fin, const void* fbase, void* fout,
                         double beta, int mode) {
    switch (v.tile) {
        case 128: return tile_launch_if_fits<T, S, MAXF, DEV, 128>(v, st, fin, fbase, fout, beta, mode);
        case 256: return tile_launch_if_fits<T, S, MAXF, DEV, 256>(v, st, fin, fbase, fout, beta, mode);
        case 512: return tile_launch_if_fits<T, S, MAXF, DEV, 512>(v, st, fin, fbase, fout, beta, mode);
        case 1024: return tile_launch_if_fits<T, S, MAXF, DEV, 1024>(v, st, fin, fbase, fout, beta, mode);
    }
    return fail(FVLBM_ERR_ARG, "unsupported tile size %d", v.tile);
}

template <typename T, typename S, bool DEV>
static int stage_t(const DevView& v, cudaStream_t st, const void* fin, const void* fbase, void* fout,
                   double beta, int mode, void* const* ev) {
    if (ev) cudaEventRecord((cudaEvent_t)ev[0], st);
    if (v.strategy == STRATEGY_TILE) {
        int rc = v.maxf == 4 ? tile_dispatch<T, S, 4, DEV>(v, st, fin, fbase, fout, beta, mode)
                             : tile_dispatch<T, S, 8, DEV>(v, st, fin, fbase, fout, beta, mode);
        if (rc) return rc;
        if (ev) {
            cudaEventRecord((cudaEvent_t)ev[1], st);
            cudaEventRecord((cudaEvent_t)ev[2], st);
        }
        return check_launch("fused stage kernel");
    }
    const int bs = v.block > 0 ? v.block : 256;   // smaller blocks spread small meshes over all SMs
    const unsigned g = grid_of(v.n_cell, bs), gg = grid_of(v.n_grad, bs);
    const S *in = (const S*)fin, *base = (const S*)fbase;
    bool lanes = false;
    if constexpr (sizeof(T) == 8) {
        // FP64: four lanes per cell until the SMs' quarters have work enough without, 198k cells of
        // four slots or 114k of eight (us per stage, lanes / a thread per cell: quads 16k 16.7 / 20.6,
        // 109k 59.5 / 66.9, 194k 100.0 / 102.2, 250k 129.5 / 129.1; triangles 180k 70.9 / 72.2,
        // 205k 80.8 / 80.0, 259k 104.5 / 100.9; polygons 116k 85.1 / 88.7, 160k 129.7 / 120.2).
        // A boundary face, whose ghost values a thread forms four times as long, outweighs eight
        // cells (0.06 of them per cell: 246k 139.6 / 143.8, 369k 203.3 / 205.2; 0.13: 410k 247.9 / 256.6;
        // 0.25: 768k 519 / 547)
        lanes = v.n_grad - 8 * v.n_bface < (v.maxf == 4 ? 1300 : 750) * (int64_t)v.sms;
        if (lanes) {
            auto kern = v.maxf == 4 ? face_values_pairs_kernel<4> : face_values_pairs_kernel<8>;
            kern<<<grid_of(4 * v.n_grad, 256), 256, 0, st>>>(v, in);
        }
    }
    if (!lanes) {
        auto kern = v.maxf == 4 ? face_values_kernel<T, S, 4, DEV> : face_values_kernel<T, S, 8, DEV>;
        kern<<<gg, bs, 0, st>>>(v, in);
    }
    if (ev) cudaEventRecord((cudaEvent_t)ev[1], st);
    auto kern = v.maxf == 4 ? update_kernel<T, S, 4, DEV> : update_kernel<T, S, 8, DEV>;
    kern<<<g, bs, 0, st>>>(v, in, base, (S*)fout, (T)beta, mode);
    if (ev) cudaEventRecord((cudaEvent_t)ev[2], st);
    return check_launch("stage kernels");
}

}  // namespace fvlbm
