// The resident stage loop: many time steps of a small solver in one launch.
//
// A mesh of a few thousand to some 60,000 cells gives every SM one tile or
// less, and a stage launched by itself is then a chain of latencies: the launch,
// the tile's record, its halo list, its geometry, its state.  Here every tile's
// CTA stays on the GPU for all the steps of the call.  Links and geometry stay
// in registers, the tile's own state in registers and shared memory; a stage
// exchanges only the halo: each cell's new state is written to the state
// buffer in global memory (L2), the CTA publishes the number of stages it has
// finished, and a thread that needs a halo cell waits for the counter of the
// tile that owns it.  There is no grid-wide barrier: a tile waits for its
// neighbours only.
//
// Order.  A stage reads one of the two state buffers and writes the other.  A
// tile enters stage s after every tile that owns one of its halo cells has
// finished stage s - 1 (2-ring neighbourhood is symmetric, so these are also
// the tiles that read this tile's cells): what it reads is written, and what it
// overwrites at the end of stage s, the input of stage s - 1, has been read.
// All CTAs are on the GPU at once (a cooperative launch; the set-up checks that
// they fit), so every wait ends; should one not, it gives up after a bounded
// number of polls, sets flag[1] and the kernel returns.
//
// The arithmetic is that of the fused stage kernel, value by value.
#pragma once

#include "fvlbm_stage.cuh"

namespace fvlbm {

constexpr int RES_POLLS = 1 << 22;   // of about half a microsecond: seconds, against microseconds of waiting

__device__ __forceinline__ uint32_t load_acquire(const uint32_t* p) {
    uint32_t x;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(p) : "memory");
    return x;
}
__device__ __forceinline__ void store_release(uint32_t* p, uint32_t x) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(x) : "memory");
}
// Waits until *p has reached `target` (counters wrap).
__device__ __forceinline__ bool wait_for(const uint32_t* p, uint32_t target) {
    for (int i = 0; i < RES_POLLS; i++)
        if ((int32_t)(load_acquire(p) - target) >= 0) return true;
    return false;
}

// The moving directions of cell i, past L1 (another SM may just have written them).
template <typename S> struct HaloCell {
    template <typename T, int LS, typename V>
    static __device__ __forceinline__ void stage(const void* fin, uint32_t i, const DevView&, int, V* fs) {
        const V* p = CellIO<S>::pairs(fin, i);
        V x[CellIO<S>::UNITS];
#pragma unroll
        for (int u = 0; u < CellIO<S>::UNITS; u++) x[u] = __ldcg(p + u * BLK);
#pragma unroll
        for (int u = 0; u < CellIO<S>::UNITS; u++) fs[u * LS] = x[u];
    }
    template <typename T> static __device__ __forceinline__ T rest(const void* fin, uint32_t i, const DevView&, int) {
        return (T)__ldcg(CellIO<S>::rest(fin, i));
    }
};
template <typename H> struct HaloSplit {
    template <typename T> static __device__ __forceinline__ void decode(const void* fin, uint32_t i, const DevView& v, int inst, T* f) {
        const uint4 h = __ldcg(CellIO<H>::head(fin, i));
        const uint2 t = __ldcg(CellIO<H>::tail(fin, i));
        CellIO<H>::template decode<T>(h, t, v.inst[inst >= 0 ? inst : v.grp[i]], f);
    }
    template <typename T, int LS, typename V>
    static __device__ __forceinline__ void stage(const void* fin, uint32_t i, const DevView& v, int inst, V* fs) {
        T f[FVLBM_Q];
        decode(fin, i, v, inst, f);
#pragma unroll
        for (int h = 0; h < 2; h++)
            store_quad(fs + h * LS, LS, Quad<T>{{f[dir_a(2 * h)], f[dir_b(2 * h)], f[dir_a(2 * h + 1)], f[dir_b(2 * h + 1)]}});
    }
    template <typename T> static __device__ __forceinline__ T rest(const void* fin, uint32_t i, const DevView& v, int inst) {
        T f[FVLBM_Q];
        decode(fin, i, v, inst, f);
        return f[0];
    }
};
template <> struct HaloCell<__half> : HaloSplit<__half> {};
template <> struct HaloCell<__nv_bfloat16> : HaloSplit<__nv_bfloat16> {};

// NS stages per step with factors beta (multistage schemes; NS = 1: Euler), or AB2.
template <typename T, typename S, int MAXF, bool DEV, int TILE, bool AB2>
__global__ void __launch_bounds__(TILE, resident_threads(sizeof(T)) / TILE)
    resident_kernel(DevView v, ResView r, int ns, int64_t stages, uint32_t epoch, int ab2_started) {
    typedef TileDims<TILE, MAXF, sizeof(T)> D;
    typedef typename Vec2<T>::type T2;
    typedef typename Vec16<T>::type V;
    constexpr int LS = D::LS, ROWS = D::ROWS;
    constexpr int SU = 8 / Vec16<T>::N;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* fs = (V*)smem_raw;         // [SU][LS]            moving directions of the local cells
    V* tab = fs + SU * LS;        // [QUAD_UNITS][ROWS]  face table
    const uint32_t t = blockIdx.x;
    const TileRec R = r.tiles[t];
    const int l = threadIdx.x, nt = R.nt, n2 = R.nt + R.n1, inst = R.inst;
    const bool mine = l < nt;
    const uint32_t gl = mine ? (uint32_t)(R.c0 + l) : l < n2 ? (uint32_t)r.halo[R.h0 + (l - nt)] : (uint32_t)R.c0;

    // what stays for the whole launch
    uint32_t d[MAXF];
    T2 c[MAXF], m[MAXF], n[MAXF];
    const GeoRef<T, MAXF> G(v.geo, gl);
    bool edge = false;
    if (l < n2) {
        if (mine) {
            load_links<MAXF>(r.link, gl, d);
        } else {
#pragma unroll
            for (int u = 0; u < MAXF / 4; u++) {
                const uint4 x = r.r1link[u * r.n_r1 + R.q0 + (l - nt)];
                d[4 * u] = x.x;
                d[4 * u + 1] = x.y;
                d[4 * u + 2] = x.z;
                d[4 * u + 3] = x.w;
            }
        }
        G.load(GEO_LSQ, c);
        G.load(GEO_MID, m);
        if (mine) G.load(GEO_FACE, n);
#pragma unroll
        for (int k = 0; k < MAXF; k++) edge |= link_boundary(d[k]);
    }
    const InstParam& P = v.inst[inst >= 0 ? inst : v.grp[gl]];
    T f[FVLBM_Q], base[FVLBM_Q], rp[FVLBM_Q];
#pragma unroll
    for (int a = 0; a < FVLBM_Q; a++) f[a] = rp[a] = T(0);
    if (mine) {
        CellIO<S>::template load<T, DEV>(v.fa, gl, P, f);
        if (AB2 && ab2_started) load_history(v, gl, rp);
    }

    int k = 0;            // stage of the step
    int other = 0;        // 0: fa -> fb, 1: fb -> fa
    bool first = AB2 && !ab2_started;
    for (int64_t s = 0; s < stages; s++) {
        const void* fin = other ? v.fb : v.fa;
        void* fout = other ? v.fa : v.fb;
        other ^= 1;
        if (k == 0) {
#pragma unroll
            for (int a = 0; a < FVLBM_Q; a++) base[a] = f[a];
        }
        // own cells to shared memory (all reads of the last stage's are past its
        // second barrier), then the halo
        Pair<T> fp[4];
        to_pairs(f, fp);
        if (mine) {
#pragma unroll
            for (int h = 0; h < 2; h++)
                store_quad(fs + h * (SU / 2) * LS + l, LS,
                           Quad<T>{{f[dir_a(2 * h)], f[dir_b(2 * h)], f[dir_a(2 * h + 1)], f[dir_b(2 * h + 1)]}});
        }
        int late = 0;
        T f0 = f[0];
        for (int e = l; e < R.nh; e += TILE) {
            if (s > 0 && !wait_for(r.done + (size_t)r.owner[R.h0 + e] * RES_STRIDE, epoch + (uint32_t)s)) {
                late = 1;
                break;
            }
            HaloCell<S>::template stage<T, LS>(fin, (uint32_t)r.halo[R.h0 + e], v, inst, fs + nt + e);
        }
        if (__syncthreads_or(late)) {
            if (late) v.flag[1] = 1;
            return;
        }
        if (l < n2) {
            if (!mine) {
                // a 1-ring cell: its state from shared memory (and f_0, for its boundary
                // faces, from its owner, whose counter the CTA has seen)
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const Quad<T> q = load_quad(fs + h * (SU / 2) * LS + l, LS);
                    fp[2 * h] = make_pair2(q.v[0], q.v[1]);
                    fp[2 * h + 1] = make_pair2(q.v[2], q.v[3]);
                }
                if (edge) f0 = HaloCell<S>::template rest<T>(fin, gl, v, inst);
            }
            tile_faces<T, DEV, MAXF, TILE>(v, d, gl, f0, fp, fs, tab, l, mine, [&](int q) { return c[q]; },
                                           [&](int q) { return m[q]; }, [&](int q) { return G.get(GEO_FACE, q); });
        }
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
            if (!update_values<T, DEV>(P, f, fp, fx, base, rp, beta, mode, out)) *v.flag = 1;
            CellIO<S>::template store_rounded<T, DEV>(fout, gl, P, out);
#pragma unroll
            for (int a = 0; a < FVLBM_Q; a++) f[a] = out[a];
        }
        first = false;
        k = k + 1 == ns ? 0 : k + 1;
        __syncthreads();
        if (l == 0) {
            __threadfence();
            store_release(r.done + (size_t)t * RES_STRIDE, epoch + (uint32_t)s + 1);
        }
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
