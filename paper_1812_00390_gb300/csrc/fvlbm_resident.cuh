// The resident stage loop: many time steps of a small solver in one launch.
//
// A mesh of a few hundred to some 100,000 cells gives every SM a few tiles or
// less, and a stage launched by itself is then a chain of latencies: the launch,
// the tile's record, its halo list, its geometry, its state.  Here every tile's
// CTA stays on the GPU for all the steps of the call.  Links stay in registers,
// geometry in shared memory (FP32; FP64 in registers, and with four tiles per SM it
// is read again), the tile's own state in both; only the halo moves between
// stages, through an exchange buffer in global memory (L2).
//
// Exchange.  A cell's new state is written as 16-byte units of three data
// words and one tag word, the number of the stage, each unit one 128-bit
// store that is seen whole or not at all.  Who needs the cell reads its units
// until all carry the tag it waits for: the data are their own signal, with no
// fence, no separate flag and no grid-wide barrier, so that a stage waits for one
// store and one load to cross the chip.  (Measured on a 128^2 cavity, FP32: with
// a counter per tile, stored with release after the data and polled with
// acquire, a stage took 4.46 us, of which 2.3 us were the fence and the polling.)
// Two sets of units alternate.  A tile overwrites at the end of stage s what it
// wrote at the end of stage s - 2; it does so after it has received the cells
// that its neighbours wrote at the end of stage s - 1, which they did after
// reading that older set (the two-ring neighbourhood is symmetric: who reads
// from a tile is read by it).
//
// All CTAs are on the GPU at once (a cooperative launch; the set-up checks that
// they fit), so every wait ends; should one not, it gives up after r.polls polls,
// sets flag[1] and the kernel returns, as do the launches queued behind it.
//
// The first stage of a launch reads its halo from the state buffer, and the
// last one writes the state buffer instead of the exchange buffer: a launch has
// at least two stages, so that every halo has been read by then.
//
// The arithmetic is that of the stage kernels, value by value, in every precision.
//
// Measured, us per stage, here / a launch per stage: 2,048 cells FP32 1.6 / 3.9;
// 128^2 cavity FP32 2.0 / 4.8; 60k-cell cylinder FP32 3.3 / 5.8, FP16 4.1 / 6.2; 12k
// polygons 2.5 / 6.9; 512 cells FP64 5.5 / 16.7, 4,096 7.0 / 18.6.  (Where the exchange buffer
// lies in memory moves these by some 1%.)
#pragma once

#include "fvlbm_stage.cuh"

namespace fvlbm {

__device__ __forceinline__ uint4 load_unit(const uint4* p) {
    uint64_t lo, hi;
    asm volatile("{ .reg .b128 x; ld.relaxed.gpu.global.b128 x, [%2]; mov.b128 {%0, %1}, x; }"
                 : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
    return make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
}
__device__ __forceinline__ void store_unit(uint4* p, uint32_t a, uint32_t b, uint32_t c, uint32_t tag) {
    const uint64_t lo = (uint64_t)b << 32 | a, hi = (uint64_t)tag << 32 | c;
    asm volatile("{ .reg .b128 x; mov.b128 x, {%1, %2}; st.relaxed.gpu.global.b128 [%0], x; }"
                 ::"l"(p), "l"(lo), "l"(hi) : "memory");
}

// Cell `i` in one set of the exchange buffer (units `stride` apart): W words of data in W / 3 units.
template <int W>
__device__ __forceinline__ bool take_cell(const uint4* p, int64_t stride, uint32_t tag, int polls, uint32_t* w) {
    for (int it = 0;; it++) {   // the first poll is free of the limit's test
        bool ok = true;
#pragma unroll
        for (int u = 0; u < W / 3; u++) {
            const uint4 x = load_unit(p + u * stride);
            w[3 * u] = x.x;
            w[3 * u + 1] = x.y;
            w[3 * u + 2] = x.z;
            ok &= x.w == tag;
        }
        if (ok) return true;
        if (it >= polls) return false;
    }
}
template <int W> __device__ __forceinline__ void give_cell(uint4* p, int64_t stride, uint32_t tag, const uint32_t* w) {
#pragma unroll
    for (int u = 0; u < W / 3; u++) store_unit(p + u * stride, w[3 * u], w[3 * u + 1], w[3 * u + 2], tag);
}

// The words of a cell in the exchange buffer: nine FP32 values, or the split
// format's six words.
template <typename S> struct Wire {
    static constexpr int W = FVLBM_Q;
    static __device__ __forceinline__ void pack(const InstParam&, const float* f, uint32_t* w) {
#pragma unroll
        for (int a = 0; a < FVLBM_Q; a++) w[a] = __float_as_uint(f[a]);
    }
    static __device__ __forceinline__ void unpack(const InstParam&, const uint32_t* w, float* f) {
#pragma unroll
        for (int a = 0; a < FVLBM_Q; a++) f[a] = __uint_as_float(w[a]);
    }
};
template <typename H> struct WireSplit {
    static constexpr int W = 6;
    // f becomes what the stored words stand for
    static __device__ __forceinline__ void pack(const InstParam& P, float* f, uint32_t* w) {
        uint4 h;
        uint2 t;
        CellIO<H>::template encode<float>(P, f, h, t);
        w[0] = h.x;
        w[1] = h.y;
        w[2] = h.z;
        w[3] = h.w;
        w[4] = t.x;
        w[5] = t.y;
        unpack(P, w, f);
    }
    static __device__ __forceinline__ void unpack(const InstParam& P, const uint32_t* w, float* f) {
        CellIO<H>::template decode<float>(make_uint4(w[0], w[1], w[2], w[3]), make_uint2(w[4], w[5]), P, f);
    }
};
template <> struct Wire<__half> : WireSplit<__half> {};
template <> struct Wire<__nv_bfloat16> : WireSplit<__nv_bfloat16> {};

template <typename T> __device__ __forceinline__ T stage_beta(int ns, int k) {
    if (ns == 1) return T(1);
    if (ns == 2) return k == 0 ? T(0.5) : T(1);
    return k == 0 ? T(0.25) : k == 1 ? T(1.0 / 3.0) : k == 2 ? T(0.5) : T(1);
}

// Deviation modes: a thread per tile and 1-ring cell, FP32.  Multistage
// schemes with ns stages per step (1: Euler), or AB2.  What does not wait for
// the halo, the own cells' collision term, is done before it is taken where a CTA
// has the SM to itself (EARLY); with several per SM it would
// hold registers that are short, and the other CTAs fill the wait.  Geometry and the step's first state sit in shared memory, each
// thread's own.
template <typename S, int MAXF, int TILE, int CTAS, bool AB2>
__global__ void __launch_bounds__(TILE, CTAS)
    resident_kernel(DevView v, ResView r, int ns, int64_t stages, uint32_t epoch, int ab2_started) {
    typedef float T;
    typedef ResDims<TILE, MAXF, sizeof(T), CTAS> D;
    typedef float2 T2;
    typedef float4 V;
    constexpr bool DEV = true;
    constexpr int LS = D::LS, ROWS = D::ROWS, W = Wire<S>::W;
    constexpr int GU = GeoRef<T, MAXF>::UNITS;
    constexpr bool EARLY = CTAS == 1, SHARED = D::GEO_SHARED;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* fs = (V*)smem_raw;         // [2][LS]       moving directions of the local cells
    V* tab = fs + 2 * LS;         // [ROWS]        face table
    V* sgeo = tab + ROWS;         // [3 GU][TILE]  geometry of the gradient cells
    V* sbase = sgeo + (SHARED ? 3 * GU * TILE : 0);   // [2][TILE]  state the step began with
    float* sbase0 = (float*)(sbase + 2 * TILE);   // [TILE]
    const int gone = *(volatile int32_t*)(v.flag + 1);   // a launch before gave up
    const TileRec R = r.tiles[blockIdx.x];
    const int l = threadIdx.x, nt = R.nt, n2 = R.nt + R.n1, n_ring2 = R.nh - R.n1, inst = R.inst;
    const bool mine = l < nt, ring1 = !mine && l < n2;
    const uint32_t gl = ring1 ? (uint32_t)r.halo[R.h0 + (l - nt)] : (uint32_t)(R.c0 + (mine ? l : 0));

    // what stays for the whole launch
    uint32_t d[MAXF];
    const GeoRef<T, MAXF> G(v.geo, gl);
    if (mine) {
        load_links<MAXF>(r.link, gl, d);
    } else if (ring1) {
#pragma unroll
        for (int u = 0; u < MAXF / 4; u++) {
            const uint4 x = r.r1link[u * r.n_r1 + R.q0 + (l - nt)];
            d[4 * u] = x.x;
            d[4 * u + 1] = x.y;
            d[4 * u + 2] = x.z;
            d[4 * u + 3] = x.w;
        }
    }
    if (SHARED && l < n2) {
#pragma unroll
        for (int u = 0; u < 3 * GU; u++) sgeo[u * TILE + l] = G.g[u * BLK];
    }
    auto geo = [&](int vec, int k) -> T2 {
        if (!SHARED) return G.get(vec, k);
        const float2* p = (const float2*)(sgeo + (vec * GU + k / 2) * TILE + threadIdx.x);
        return p[k % 2];
    };
    auto geo_all = [&](int vec, T2* out) {   // in 16-byte loads: no bank conflict
#pragma unroll
        for (int u = 0; u < GU; u++) {
            const V q = SHARED ? sgeo[(vec * GU + u) * TILE + threadIdx.x] : G.g[(vec * GU + u) * BLK];
            out[2 * u] = make_float2(q.x, q.y);
            out[2 * u + 1] = make_float2(q.z, q.w);
        }
    };
    const InstParam& P = v.inst[inst >= 0 ? inst : v.grp[gl]];
    const Relax<T> relax(P);
    T f[FVLBM_Q], rp[FVLBM_Q];
#pragma unroll
    for (int a = 0; a < FVLBM_Q; a++) f[a] = rp[a] = T(0);
    if (l < n2) CellIO<S>::template load<T, DEV>(v.fa, gl, P, f);
    if (AB2 && mine && ab2_started) load_history(v, gl, rp);

    auto quad = [](const T* q, int h) {
        return Quad<T>{{q[dir_a(2 * h)], q[dir_b(2 * h)], q[dir_a(2 * h + 1)], q[dir_b(2 * h + 1)]}};
    };
    auto to_shared = [&](int x, const T* q) {
        store_quad(fs + x, LS, quad(q, 0));
        store_quad(fs + LS + x, LS, quad(q, 1));
    };
    auto lsq = [&](int q) { return geo(GEO_LSQ, q); };
    auto face = [&](int q) { return geo(GEO_FACE, q); };
    if (__syncthreads_or(gone)) return;
    int k = 0;            // stage of the step
    bool first = AB2 && !ab2_started;
    for (int64_t s = 0; s < stages; s++) {
        const uint4* from = r.xchg + (s & 1) * (W / 3) * v.np;
        const uint32_t tag = epoch + (uint32_t)s;
        // the local cells' state into shared memory (every read of the last stage's
        // is behind its second barrier): own cells, 1-ring cells by the thread that
        // computes their gradient, 2-ring cells by all
        int late = 0;
        T col[FVLBM_Q];
        Pair<T> fp[4], gx[4], gy[4];
        if (mine) {
            to_shared(l, f);
            if (!AB2 && k == 0) {
                store_quad(sbase + l, TILE, quad(f, 0));
                store_quad(sbase + TILE + l, TILE, quad(f, 1));
                sbase0[l] = f[0];
            }
            if (EARLY) collision<T, DEV>(f, col);
        } else if (ring1) {
            if (s > 0) {
                uint32_t w[W];
                late = !take_cell<W>(from + gl, v.np, tag, r.polls, w);
                Wire<S>::unpack(P, w, f);
            }
            to_shared(l, f);
        }
        for (int e = l; e < n_ring2; e += TILE) {
            const uint32_t i = (uint32_t)__ldg(r.halo + R.h0 + R.n1 + e);
            const InstParam& Pi = v.inst[inst >= 0 ? inst : v.grp[i]];
            T q[FVLBM_Q];
            if (s > 0) {
                uint32_t w[W];
                late |= !take_cell<W>(from + i, v.np, tag, r.polls, w);
                Wire<S>::unpack(Pi, w, q);
            } else {
                CellIO<S>::template load<T, DEV>(v.fa, i, Pi, q);
            }
            to_shared(n2 + e, q);
        }
        if (__syncthreads_or(late)) {
            if (late) v.flag[1] = 1;
            return;
        }
        if (l < n2) {
            to_pairs(f, fp);
            T2 c[MAXF], m[MAXF];
            geo_all(GEO_LSQ, c);
            tile_faces<T, DEV, MAXF, TILE>(d, fp, gx, gy, fs, tab, l, [&](int q) { return c[q]; },
                                           [&](int q) { return m[q]; }, [&] { geo_all(GEO_MID, m); }, [&] {
                tile_boundary<T, DEV, MAXF, TILE, true>(v.bc, v.bctag, d, gl, f[0], fp, gx, gy, tab, l, mine, lsq, face);
            });
        }
        __syncthreads();
        if (mine) {
            Pair<T> fx[4];
#pragma unroll
            for (int p = 0; p < 4; p++) fx[p] = make_pair2(T(0), T(0));
            const uint32_t used = warp_slots<MAXF>(d);
            T2 n[MAXF];
            geo_all(GEO_FACE, n);
#pragma unroll
            for (int q = 0; q < MAXF; q++) {
                if (q >= 3 && !((used >> q) & 1u)) continue;
                add_flux<T, DEV>(d[q], n[q], load_quad(tab + q * TILE + l, ROWS),
                                 load_quad(tab + link_row(d[q]), ROWS), fp, fx);
            }
            T out[FVLBM_Q], base[FVLBM_Q];
            if (!EARLY) collision<T, DEV>(f, col);
            if (!AB2) {
                const Quad<T> b0 = load_quad(sbase + l, TILE), b1 = load_quad(sbase + TILE + l, TILE);
                const Pair<T> bp[4] = {make_pair2(b0.v[0], b0.v[1]), make_pair2(b0.v[2], b0.v[3]),
                                       make_pair2(b1.v[0], b1.v[1]), make_pair2(b1.v[2], b1.v[3])};
                from_pairs(bp, base);
                base[0] = sbase0[l];
            }
            const int mode = AB2 ? (first ? MODE_AB2_FIRST : MODE_AB2) : MODE_RK;
            const bool ok = advance<T, DEV>(relax, f, col, fx, base, rp, stage_beta<T>(ns, k), mode, out);
            if (s + 1 < stages) {
                uint32_t w[W];
                Wire<S>::pack(P, out, w);
                give_cell<W>(r.xchg + ((s + 1) & 1) * (W / 3) * v.np + gl, v.np, tag + 1, w);
            } else {
                CellIO<S>::template store<T, DEV>(v.fa, gl, P, out);
            }
            if (!ok) *v.flag = 1;
#pragma unroll
            for (int a = 0; a < FVLBM_Q; a++) f[a] = out[a];
        }
        first = false;
        k = k + 1 == ns ? 0 : k + 1;
    }
    if (AB2 && mine) store_history(v, gl, rp);
}

// FP64: four lanes per tile and 1-ring cell, one for each pair of directions.
// GB300 has one FP64 unit per SM quarter, which takes 64 cycles for a warp's
// instruction whatever its active lanes, so a tile that gives each quarter less than
// a warp of cells leaves it idle most of the time (512 cells, one thread per
// cell: 12.9 us per stage, of which 12,500 cycles the gradients and 8,100 the
// update).  With a pair per lane a warp's 8 cells take a quarter of the instructions,
// and the moments are formed by two rounds of shuffles, in the order of
// moments() (bitwise the same).  A lane's geometry stays in registers; e.n of its
// pair is formed once.  In the exchange buffer a lane's two units carry its two
// values and the two halves of f_0.
template <int MAXF, int TILE, bool AB2>
__global__ void __launch_bounds__(RES_LANES_FP64* TILE, 1)
    resident_pairs_kernel(DevView v, ResView r, int ns, int64_t stages, uint32_t epoch, int ab2_started) {
    typedef double T;
    typedef TileDims<TILE, MAXF, sizeof(T)> D;
    constexpr int LS = D::LS, ROWS = D::ROWS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2* fs = (double2*)smem_raw;   // [LS][4]    pairs of the local cells
    double* tab = (double*)(fs + 4 * LS);   // [ROWS][4]  face table
    const int gone = *(volatile int32_t*)(v.flag + 1);   // a launch before gave up
    const TileRec R = r.tiles[blockIdx.x];
    const int x = threadIdx.x >> 2, p = threadIdx.x & 3, nt = R.nt, n2 = R.nt + R.n1, n_ring2 = R.nh - R.n1,
              inst = R.inst;
    const bool mine = x < nt, ring1 = !mine && x < n2;
    const uint32_t gl = ring1 ? (uint32_t)r.halo[R.h0 + (x - nt)] : (uint32_t)(R.c0 + (mine ? x : 0));

    // what stays for the whole launch
    uint32_t d[MAXF];
    double2 c[MAXF], m[MAXF];
    double en[MAXF];
    const GeoRef<T, MAXF> G(v.geo, gl);
#pragma unroll
    for (int k = 0; k < MAXF; k++) d[k] = (uint32_t)LK_NONE << LINK_KIND_SHIFT;
    if (mine) {
        load_links<MAXF>(r.link, gl, d);
    } else if (ring1) {
#pragma unroll
        for (int u = 0; u < MAXF / 4; u++) {
            const uint4 q = r.r1link[u * r.n_r1 + R.q0 + (x - nt)];
            d[4 * u] = q.x;
            d[4 * u + 1] = q.y;
            d[4 * u + 2] = q.z;
            d[4 * u + 3] = q.w;
        }
    }
    if (x < n2) {
#pragma unroll
        for (int k = 0; k < MAXF; k++) {
            c[k] = G.get(GEO_LSQ, k);
            m[k] = G.get(GEO_MID, k);
            const double2 n = G.get(GEO_FACE, k);
            en[k] = p == 0 ? n.x : p == 1 ? n.y : p == 2 ? n.x + n.y : n.y - n.x;
        }
    }
    const uint32_t edges = boundary_mask<MAXF>(d);
    const bool edge = edges != 0;
    uint32_t used = 7u;
#pragma unroll
    for (int k = 3; k < MAXF; k++)
        if (link_kind(d[k]) != LK_NONE) used |= 1u << k;
    used = __reduce_or_sync(0xFFFFFFFFu, used);
    const bool warp_mine = __any_sync(0xFFFFFFFFu, mine), warp_ring_edge = __any_sync(0xFFFFFFFFu, ring1 && edge);
    const InstParam& P = v.inst[inst >= 0 ? inst : v.grp[gl]];
    const Relax<T> relax(P);
    const double w = lane_weight(p);
    double f0 = 0, fa = 0, fb = 0, b0 = 0, ba = 0, bb = 0, rp0 = 0, rpa = 0, rpb = 0;
    const int ia = dir_a(0) * (p == 0) + dir_a(1) * (p == 1) + dir_a(2) * (p == 2) + dir_a(3) * (p == 3);
    const int ib = dir_b(0) * (p == 0) + dir_b(1) * (p == 1) + dir_b(2) * (p == 2) + dir_b(3) * (p == 3);
    auto load_state = [&](uint32_t i, double& q0, double& qa, double& qb) {
        const double2 q = CellIO<double>::pairs(v.fa, i)[p * BLK];
        qa = q.x;
        qb = q.y;
        q0 = *CellIO<double>::rest(v.fa, i);
    };
    if (x < n2) load_state(gl, f0, fa, fb);
    double* hist = (double*)v.rprev;
    if (AB2 && mine && ab2_started) {
        rp0 = hist[gl];
        rpa = hist[ia * v.np + gl];
        rpb = hist[ib * v.np + gl];
    }

    if (__syncthreads_or(gone)) return;
    int k = 0;            // stage of the step
    bool first = AB2 && !ab2_started;
    for (int64_t s = 0; s < stages; s++) {
        const uint4* from = r.xchg + (s & 1) * 8 * v.np;
        const uint32_t tag = epoch + (uint32_t)s;
        if (k == 0) {
            b0 = f0;
            ba = fa;
            bb = fb;
        }
        // take the lane's pair (and f_0) of cell i
        auto take = [&](uint32_t i, double& q0, double& qa, double& qb) {
            uint32_t u[6];
            const bool ok = take_cell<6>(from + ((size_t)i * 8 + p * 2), 1, tag, r.polls, u);
            qa = __hiloint2double((int)u[1], (int)u[0]);
            qb = __hiloint2double((int)u[4], (int)u[3]);
            q0 = __hiloint2double((int)u[5], (int)u[2]);
            return ok;
        };
        // ghost differences: the gradient's start, and the rows of the face table that
        // only this cell reads
        double gax = 0, gay = 0, gbx = 0, gby = 0;
        auto boundary = [&](double rho, double ux, double uy, double qa, double qb) {
            lane_boundary<MAXF>(p, d, v.bc, fa, fb, rho, ux, uy, qa, qb, gax, gay, gbx, gby,
                                [&](int q) { return v.bctag[(int64_t)gl * MAXF + q]; },
                                [&](int q) { return G.get(GEO_LSQ, q); }, [&](int q) { return G.get(GEO_FACE, q); },
                                [&](int q, double z) { tab[(q * TILE + x) * 4 + p] = z; },
                                [&](int, uint32_t dq, double z) {
                                    if (mine) tab[link_row(dq) * 4 + p] = z;
                                });
        };
        int late = 0;
        double col0 = 0, cola = 0, colb = 0, c1 = 0, c2 = 0;
        if (mine) fs[x * 4 + p] = make_double2(fa, fb);
        if (warp_mine) {   // what needs the own state only, before the halo is there
            double rho, ux, uy, qa, qb, q0;
            lanes_moments(p, f0, fa, fb, rho, ux, uy);
            lane_eq(p, ux, uy, qa, qb, q0);
            c1 = stage_beta<T>(ns, k) * relax.dt;
            c2 = c1 * relax.inv_tau;
            if (mine) {
                const double rw = rho * w;
                col0 = fma(rho * (4.0 / 9.0), q0, -f0);
                cola = fma(rw, qa, -fa);
                colb = fma(rw, qb, -fb);
                if (edge) boundary(rho, ux, uy, qa, qb);
            }
        }
        if (ring1) {
            if (s > 0) late = !take(gl, f0, fa, fb);
            fs[x * 4 + p] = make_double2(fa, fb);
        }
        if (warp_ring_edge) {   // 1-ring cells' boundary faces
            double rho, ux, uy, qa, qb, q0;
            lanes_moments(p, f0, fa, fb, rho, ux, uy);
            lane_eq(p, ux, uy, qa, qb, q0);
            if (ring1 && edge) boundary(rho, ux, uy, qa, qb);
        }
        for (int e = x; e < n_ring2; e += TILE) {
            const uint32_t i = (uint32_t)__ldg(r.halo + R.h0 + R.n1 + e);
            double h0, ha, hb;
            if (s > 0) late |= !take(i, h0, ha, hb);
            else load_state(i, h0, ha, hb);
            fs[(n2 + e) * 4 + p] = make_double2(ha, hb);
        }
        if (__syncthreads_or(late)) {
            if (late) v.flag[1] = 1;
            return;
        }
        if (x < n2) {
#pragma unroll
            for (int q = 0; q < MAXF; q++) {
                if (q >= 3 && !((used >> q) & 1u)) continue;
                const double2 nb = fs[(d[q] & LINK_NB_MASK) * 4 + p];
                const double da = nb.x - fa, db = nb.y - fb;
                gax = fma(c[q].x, da, gax);
                gay = fma(c[q].y, da, gay);
                gbx = fma(c[q].x, db, gbx);
                gby = fma(c[q].y, db, gby);
            }
#pragma unroll
            for (int q = 0; q < MAXF; q++) {
                if (q >= 3 && !((used >> q) & 1u)) continue;
                const uint32_t kind = link_kind(d[q]);
                if (kind == LK_FLOW || kind == LK_NONE || kind_io(kind)) {
                    const bool a = link_a_leaves(d[q], p);
                    tab[(q * TILE + x) * 4 + p] = fma(a ? gay : gby, m[q].y, fma(a ? gax : gbx, m[q].x, a ? fa : fb));
                }
            }
        }
        __syncthreads();
        if (mine) {
            double la = 0, lb = 0;
#pragma unroll
            for (int q = 0; q < MAXF; q++) {
                if (q >= 3 && !((used >> q) & 1u)) continue;
                const double out = tab[(q * TILE + x) * 4 + p], in = tab[link_row(d[q]) * 4 + p];
                const bool a = link_a_leaves(d[q], p);
                la = fma(en[q], a ? out : in, la);
                lb = fma(-en[q], a ? in : out, lb);
            }
            double o0, oa, ob;
            if (!AB2) {
                o0 = fma(c2, col0, b0);
                oa = fma(c2, cola, fma(-c1, la, ba));
                ob = fma(c2, colb, fma(-c1, lb, bb));
            } else {
                const double r0 = fma(relax.inv_tau, col0, -0.0), ra = fma(relax.inv_tau, cola, -la),
                             rb = fma(relax.inv_tau, colb, -lb);
                o0 = fma(relax.dt, first ? r0 : fma(1.5, r0, -0.5 * rp0), f0);
                oa = fma(relax.dt, first ? ra : fma(1.5, ra, -0.5 * rpa), fa);
                ob = fma(relax.dt, first ? rb : fma(1.5, rb, -0.5 * rpb), fb);
                rp0 = r0;
                rpa = ra;
                rpb = rb;
            }
            f0 = o0;
            fa = oa;
            fb = ob;
            if (s + 1 < stages) {
                const uint32_t u[6] = {(uint32_t)__double2loint(fa), (uint32_t)__double2hiint(fa), (uint32_t)__double2loint(f0),
                                       (uint32_t)__double2loint(fb), (uint32_t)__double2hiint(fb), (uint32_t)__double2hiint(f0)};
                give_cell<6>(r.xchg + ((s + 1) & 1) * 8 * v.np + ((size_t)gl * 8 + p * 2), 1, tag + 1, u);
            } else {
                ((double2*)CellIO<double>::pairs(v.fa, gl))[p * BLK] = make_double2(fa, fb);
                if (p == 0) *(double*)CellIO<double>::rest(v.fa, gl) = f0;
            }
            if (!(finite_val(f0) && finite_val(fa) && finite_val(fb))) *v.flag = 1;
        }
        first = false;
        k = k + 1 == ns ? 0 : k + 1;
    }
    if (AB2 && mine) {
        if (p == 0) hist[gl] = rp0;
        hist[ia * v.np + gl] = rpa;
        hist[ib * v.np + gl] = rpb;
    }
}

// Launch of one kernel; with max_ctas, only how many of its CTAs fit on the GPU at once.
static int resident_launch(const void* kern, int threads, size_t smem, const DevView& v, const ResView& r, cudaStream_t st,
                           int scheme, int64_t stages, uint32_t epoch, bool ab2_started, int* max_ctas) {
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return fail(FVLBM_ERR_CUDA, "resident stage loop: %zu B shared memory: %s", smem, cudaGetErrorString(e));
    }
    if (max_ctas) {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess) {
            cudaGetLastError();
            per_sm = 0;
        }
        *max_ctas = per_sm * v.sms;
        return FVLBM_OK;
    }
    int ns = scheme == FVLBM_RK2 ? 2 : scheme == FVLBM_RK4 ? 4 : 1, started = ab2_started ? 1 : 0;
    DevView vv = v;
    ResView rr = r;
    void* args[] = {&vv, &rr, &ns, &stages, &epoch, &started};
    cudaError_t e = cudaLaunchCooperativeKernel(kern, dim3((unsigned)r.n_tiles), dim3((unsigned)threads), args, smem, st);
    // refused as a whole: the tiles do not all fit where the stream's launches run
    // (fewer SMs than the device has), or cooperative launches are not to be had there
    if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
        cudaGetLastError();
        return fail(FVLBM_ERR_UNSUPPORTED, "resident stage loop: %s", cudaGetErrorString(e));
    }
    if (e != cudaSuccess) return fail(FVLBM_ERR_CUDA, "resident stage loop: %s", cudaGetErrorString(e));
    return FVLBM_OK;
}

// The kernel of a tile size (`ctas` of them per SM), slot count and scheme.
template <typename S, int MAXF, int TILE, int CTAS>
static const void* resident_of(int scheme, int& threads, size_t& smem) {
    const bool ab2 = scheme == FVLBM_AB2;
    if constexpr (sizeof(S) == 8) {
        threads = RES_LANES_FP64 * TILE;
        smem = TileDims<TILE, MAXF, 8>::BYTES;
        return ab2 ? (const void*)resident_pairs_kernel<MAXF, TILE, true> : (const void*)resident_pairs_kernel<MAXF, TILE, false>;
    } else {
        threads = TILE;
        smem = ResDims<TILE, MAXF, 4, CTAS>::BYTES;
        return ab2 ? (const void*)resident_kernel<S, MAXF, TILE, CTAS, true>
                   : (const void*)resident_kernel<S, MAXF, TILE, CTAS, false>;
    }
}

template <typename S, int MAXF>
static int resident_m(const DevView& v, const ResView& r, cudaStream_t st, int scheme, int64_t stages, uint32_t epoch,
                      bool ab2_started, int* max_ctas) {
    const void* kern = nullptr;
    int threads = 0;
    size_t smem = 0;
    if constexpr (sizeof(S) == 8) {
        if (r.tile == RES_TILE_FP64) kern = resident_of<S, MAXF, RES_TILE_FP64, 1>(scheme, threads, smem);
    } else {
        constexpr int MORE = resident_ctas(4, MAXF);
        if (r.tile == RES_TILE / 2) kern = resident_of<S, MAXF, RES_TILE / 2, 1>(scheme, threads, smem);
        if (r.tile == RES_TILE)
            kern = r.n_tiles <= v.sms       ? resident_of<S, MAXF, RES_TILE, 1>(scheme, threads, smem)
                   : r.n_tiles <= 3 * v.sms ? resident_of<S, MAXF, RES_TILE, MORE < 3 ? MORE : 3>(scheme, threads, smem)
                                            : resident_of<S, MAXF, RES_TILE, MORE>(scheme, threads, smem);
    }
    if (!kern) return fail(FVLBM_ERR_ARG, "resident stage loop: tiles of %d cells", r.tile);
    return resident_launch(kern, threads, smem, v, r, st, scheme, stages, epoch, ab2_started, max_ctas);
}

template <typename S>
static int resident_t(const DevView& v, const ResView& r, cudaStream_t st, int scheme, int64_t stages, uint32_t epoch,
                      bool ab2_started, int* max_ctas) {
    return v.maxf == 4 ? resident_m<S, 4>(v, r, st, scheme, stages, epoch, ab2_started, max_ctas)
                       : resident_m<S, 8>(v, r, st, scheme, stages, epoch, ab2_started, max_ctas);
}

}  // namespace fvlbm
