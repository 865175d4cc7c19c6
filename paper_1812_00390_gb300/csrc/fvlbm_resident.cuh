// The resident stage loop: many time steps of a small solver in one launch.
//
// A mesh of a few hundred to some 60,000 cells gives every SM one tile or
// less, and a stage launched by itself is then a chain of latencies: the launch,
// the tile's record, its halo list, its geometry, its state.  Here every tile's
// CTA stays on the GPU for all the steps of the call.  Links and geometry stay
// in registers, the tile's own state in registers and shared memory; only the
// halo moves between stages, through an exchange buffer in global memory (L2).
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
// they fit), so every wait ends; should one not, it gives up after a bounded
// number of polls, sets flag[1] and the kernel returns.
//
// The first stage of a launch reads its halo from the state buffer, and the
// last one writes the state buffer instead of the exchange buffer: a launch has
// at least two stages, so that every halo has been read by then.
//
// The arithmetic is that of the fused stage kernel, value by value.
#pragma once

#include "fvlbm_stage.cuh"

namespace fvlbm {

constexpr int RES_POLLS = 1 << 22;   // of about half a microsecond: seconds, against microseconds of waiting

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
template <int W> __device__ __forceinline__ bool take_cell(const uint4* p, int64_t stride, uint32_t tag, uint32_t* w) {
    for (int it = 0; it < RES_POLLS; it++) {
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
    }
    return false;
}
template <int W> __device__ __forceinline__ void give_cell(uint4* p, int64_t stride, uint32_t tag, const uint32_t* w) {
#pragma unroll
    for (int u = 0; u < W / 3; u++) store_unit(p + u * stride, w[3 * u], w[3 * u + 1], w[3 * u + 2], tag);
}

// The words of a cell in the exchange buffer: nine values, or the split format's six words.
template <typename S> struct Wire {
    static constexpr int W = FVLBM_Q * sizeof(S) / 4;
    template <typename T> static __device__ __forceinline__ void pack(const InstParam&, T* f, uint32_t* w) {
#pragma unroll
        for (int a = 0; a < FVLBM_Q; a++) {
            if constexpr (sizeof(T) == 4) {
                w[a] = __float_as_uint(f[a]);
            } else {
                w[2 * a] = (uint32_t)__double2loint(f[a]);
                w[2 * a + 1] = (uint32_t)__double2hiint(f[a]);
            }
        }
    }
    template <typename T> static __device__ __forceinline__ void unpack(const InstParam&, const uint32_t* w, T* f) {
#pragma unroll
        for (int a = 0; a < FVLBM_Q; a++) {
            if constexpr (sizeof(T) == 4) f[a] = __uint_as_float(w[a]);
            else f[a] = __hiloint2double((int)w[2 * a + 1], (int)w[2 * a]);
        }
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

// Multistage schemes with ns stages per step (1: Euler), or AB2.
template <typename T, typename S, int MAXF, bool DEV, int TILE, bool AB2>
__global__ void __launch_bounds__(TILE, resident_threads(sizeof(T)) / TILE)
    resident_kernel(DevView v, ResView r, int ns, int64_t stages, uint32_t epoch, int ab2_started) {
    typedef TileDims<TILE, MAXF, sizeof(T)> D;
    typedef typename Vec2<T>::type T2;
    typedef typename Vec16<T>::type V;
    constexpr int LS = D::LS, ROWS = D::ROWS, W = Wire<S>::W;
    constexpr int SU = 8 / Vec16<T>::N;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* fs = (V*)smem_raw;         // [SU][LS]            moving directions of the local cells
    V* tab = fs + SU * LS;        // [QUAD_UNITS][ROWS]  face table
    const TileRec R = r.tiles[blockIdx.x];
    const int l = threadIdx.x, nt = R.nt, n2 = R.nt + R.n1, n_ring2 = R.nh - R.n1, inst = R.inst;
    const bool mine = l < nt, ring1 = !mine && l < n2;
    const uint32_t gl = ring1 ? (uint32_t)r.halo[R.h0 + (l - nt)] : (uint32_t)(R.c0 + (mine ? l : 0));

    // what stays for the whole launch
    uint32_t d[MAXF];
    T2 c[MAXF], m[MAXF], n[MAXF];
    const GeoRef<T, MAXF> G(v.geo, gl);
    if (mine) {
        load_links<MAXF>(r.link, gl, d);
        G.load(GEO_FACE, n);
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
    if (l < n2) {
        G.load(GEO_LSQ, c);
        G.load(GEO_MID, m);
    }
    const InstParam& P = v.inst[inst >= 0 ? inst : v.grp[gl]];
    const Relax<T> relax(P);
    T f[FVLBM_Q], base[FVLBM_Q], rp[FVLBM_Q];
#pragma unroll
    for (int a = 0; a < FVLBM_Q; a++) f[a] = rp[a] = T(0);
    if (l < n2) CellIO<S>::template load<T, DEV>(v.fa, gl, P, f);
    if (AB2 && mine && ab2_started) load_history(v, gl, rp);

    auto to_shared = [&](int x, const T* q) {
#pragma unroll
        for (int h = 0; h < 2; h++)
            store_quad(fs + h * (SU / 2) * LS + x, LS,
                       Quad<T>{{q[dir_a(2 * h)], q[dir_b(2 * h)], q[dir_a(2 * h + 1)], q[dir_b(2 * h + 1)]}});
    };
    int k = 0;            // stage of the step
    bool first = AB2 && !ab2_started;
    for (int64_t s = 0; s < stages; s++) {
        const uint4* from = r.xchg + (s & 1) * (W / 3) * v.np;
        const uint32_t tag = epoch + (uint32_t)s;
        if (k == 0) {
#pragma unroll
            for (int a = 0; a < FVLBM_Q; a++) base[a] = f[a];
        }
        // the local cells' state into shared memory (every read of the last stage's
        // is behind its second barrier): own cells, 1-ring cells by the thread that
        // computes their gradient, 2-ring cells by all
        int late = 0;
        if (ring1 && s > 0) {
            uint32_t w[W];
            late = !take_cell<W>(from + gl, v.np, tag, w);
            Wire<S>::unpack(P, w, f);
        }
        if (l < n2) to_shared(l, f);
        for (int e = l; e < n_ring2; e += TILE) {
            const uint32_t i = (uint32_t)__ldg(r.halo + R.h0 + R.n1 + e);
            const InstParam& Pi = v.inst[inst >= 0 ? inst : v.grp[i]];
            T q[FVLBM_Q];
            if (s > 0) {
                uint32_t w[W];
                late |= !take_cell<W>(from + i, v.np, tag, w);
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
        Pair<T> fp[4];
        to_pairs(f, fp);
        if (l < n2)
            tile_faces<T, DEV, MAXF, TILE>(v, d, gl, f[0], fp, fs, tab, l, mine, [&](int q) { return c[q]; },
                                           [&](int q) { return m[q]; }, [&](int q) { return G.get(GEO_FACE, q); });
        __syncthreads();
        if (mine) {
            Pair<T> fx[4];
#pragma unroll
            for (int p = 0; p < 4; p++) fx[p] = make_pair2(T(0), T(0));
            const uint32_t used = warp_slots<MAXF>(d);
#pragma unroll
            for (int q = 0; q < MAXF; q++) {
                if (q >= 3 && !((used >> q) & 1u)) continue;
                add_flux<T, DEV>(d[q], n[q], load_quad(tab + q * TILE + l, ROWS), load_quad(tab + link_row(d[q]), ROWS), fp, fx);
            }
            T out[FVLBM_Q];
            const T beta = ns == 1 ? T(1) : ns == 2 ? (k == 0 ? T(0.5) : T(1))
                         : k == 0 ? T(0.25) : k == 1 ? T(1.0 / 3.0) : k == 2 ? T(0.5) : T(1);
            const int mode = AB2 ? (first ? MODE_AB2_FIRST : MODE_AB2) : MODE_RK;
            if (!update_values<T, DEV>(relax, f, fp, fx, base, rp, beta, mode, out)) *v.flag = 1;
            if (s + 1 < stages) {
                uint32_t w[W];
                Wire<S>::pack(P, out, w);
                give_cell<W>(r.xchg + ((s + 1) & 1) * (W / 3) * v.np + gl, v.np, tag + 1, w);
            } else {
                CellIO<S>::template store<T, DEV>(v.fa, gl, P, out);
            }
#pragma unroll
            for (int a = 0; a < FVLBM_Q; a++) f[a] = out[a];
        }
        first = false;
        k = k + 1 == ns ? 0 : k + 1;
    }
    if (AB2 && mine) store_history(v, gl, rp);
}

// Launch of one instantiation; with max_ctas, only how many of its CTAs fit on the GPU at once.
template <typename T, typename S, int MAXF, bool DEV, int TILE, bool AB2>
static int resident_launch(const DevView& v, const ResView& r, cudaStream_t st, int ns, int64_t stages, uint32_t epoch,
                           bool ab2_started, int* max_ctas) {
    auto kern = resident_kernel<T, S, MAXF, DEV, TILE, AB2>;
    const size_t smem = TileDims<TILE, MAXF, sizeof(T)>::BYTES;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return fail(FVLBM_ERR_CUDA, "resident stage loop: %zu B shared memory: %s", smem, cudaGetErrorString(e));
    }
    if (max_ctas) {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, TILE, smem) != cudaSuccess) {
            cudaGetLastError();
            per_sm = 0;
        }
        *max_ctas = per_sm * v.sms;
        return FVLBM_OK;
    }
    int started = ab2_started ? 1 : 0;
    DevView vv = v;
    ResView rr = r;
    void* args[] = {&vv, &rr, &ns, &stages, &epoch, &started};
    cudaError_t e = cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)r.n_tiles), dim3(TILE), args, smem, st);
    if (e != cudaSuccess) return fail(FVLBM_ERR_CUDA, "resident stage loop: %s", cudaGetErrorString(e));
    return FVLBM_OK;
}

template <typename T, typename S, bool DEV, int MAXF, int TILE>
static int resident_scheme(const DevView& v, const ResView& r, cudaStream_t st, int scheme, int64_t stages, uint32_t epoch,
                           bool ab2_started, int* max_ctas) {
    const int ns = scheme == FVLBM_RK2 ? 2 : scheme == FVLBM_RK4 ? 4 : 1;
    if (scheme == FVLBM_AB2)
        return resident_launch<T, S, MAXF, DEV, TILE, true>(v, r, st, ns, stages, epoch, ab2_started, max_ctas);
    return resident_launch<T, S, MAXF, DEV, TILE, false>(v, r, st, ns, stages, epoch, ab2_started, max_ctas);
}

template <typename T, typename S, bool DEV>
static int resident_t(const DevView& v, const ResView& r, cudaStream_t st, int scheme, int64_t stages, uint32_t epoch,
                      bool ab2_started, int* max_ctas) {
#define FVLBM_RES(T_)                                                                                                \
    if (r.tile == T_)                                                                                                \
        return v.maxf == 4 ? resident_scheme<T, S, DEV, 4, T_>(v, r, st, scheme, stages, epoch, ab2_started, max_ctas) \
                           : resident_scheme<T, S, DEV, 8, T_>(v, r, st, scheme, stages, epoch, ab2_started, max_ctas);
    if constexpr (sizeof(T) == 4) {
        FVLBM_RES(512)
    } else {
        FVLBM_RES(32)
    }
    FVLBM_RES(64)
    FVLBM_RES(128)
    FVLBM_RES(256)
#undef FVLBM_RES
    return fail(FVLBM_ERR_ARG, "resident stage loop: %d threads per CTA", r.tile);
}

}  // namespace fvlbm
