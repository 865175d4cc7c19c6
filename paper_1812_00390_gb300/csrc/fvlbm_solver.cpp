// Solver lifecycle and the C ABI entry points that touch the GPU.
//
// fvlbm_init packs the FP64 mesh precompute into the device layout of the
// chosen precision (SoA planes [slot][cell] in the locality order), uploads it
// into one workspace, and writes Step 0 (f = f^eq).  fvlbm_step enqueues the
// stages of the time scheme (Sec. 2.3) on the solver's stream.  Everything
// that reads results back (macros, residual, mass, f) synchronises and maps
// cells back to the caller's numbering.
#include <algorithm>
#include <chrono>
#include <cstdio>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>

#include <cuda_runtime.h>

#include "fvlbm_internal.h"

namespace fvlbm {
double suggest_dt(const Mesh& M, int inst, double tau, double cfl, double umax, int scheme);
}

using namespace fvlbm;

struct fvlbm_solver {
    int device = 0;
    cudaStream_t stream = nullptr;
    int prec = FVLBM_FP64;
    int scheme = FVLBM_EULER;
    int64_t n_cell = 0;
    int32_t n_inst = 1;
    std::vector<int64_t> inst_begin;
    void* ws = nullptr;
    size_t ws_bytes = 0;
    bool own_ws = false;
    DevView v{};
    std::vector<InstParam> inst;
    bool ab2_started = false;
    // set_f reads the caller's host buffer directly (see fvlbm_host_transfer)
    bool host_can_direct = false;
    bool host_direct = false;
    // single-stage schemes on the fused stage alternate the state between
    // buf[0] and buf[1] (a tile must not overwrite cells other tiles still
    // read); v.fa is always the current state, buf[cur]
    bool pingpong = false;
    void* buf[2] = {nullptr, nullptr};
    int cur = 0;
    // the 4-stage scheme on the fused stage: a third stage buffer, so that no
    // stage writes the buffer it reads (the middle stages alternate fb, fc)
    void* fc = nullptr;
    // CUDA graphs of one step and of GRAPH_CHUNK steps, built lazily, one pair
    // per state buffer the step starts from
    cudaGraphExec_t g1[2] = {nullptr, nullptr}, gk[2] = {nullptr, nullptr};
    bool graphs_ok = true;
    int64_t direct_steps = 0;
    bool staged = false;   // a stage has been launched by itself (partitioned solve)
    // small solvers: steps run in the resident stage loop; exchange tags used so far
    bool resident = false;
    ResView res{};
    uint32_t epoch = 0;
    int64_t res_launches = 0;
    StepPath path = STEP_AUTO;
    StageCost cost;
    // who steps beside this solver (Crowd): the time at which its last long call is expected
    // to be done; number of that call; whether another solver stepped meanwhile
    bool member = false, joined = false;
    double busy_until = 0;
    uint64_t call = 0;
    double lost = 0;   // microseconds that its calls in turns took longer than overlapping
};

static constexpr int64_t GRAPH_CHUNK = 32;
// What a solver's first stage kernels take besides, for both graphs captured and
// instantiated: the host's time (eight solvers' first 600 stages 0.5 to 1 ms each), and what
// a fresh request pays while its neighbours start (requests of 2,000 steps served both
// ways: 4 to 7 ms each, of 4k quads in FP64 17).
static constexpr double GRAPH_SETUP_US = 1000;
static double request_setup_us(int prec) { return prec == FVLBM_FP64 ? 18000 : 6000; }
// stages of one resident launch (a few milliseconds)
static constexpr int64_t RESIDENT_CHUNK = 2048;

namespace {

int cuda_fail(cudaError_t e, const char* what) {
    return fail(FVLBM_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define CK(call, what)                                  \
    do {                                                \
        cudaError_t e_ = (call);                        \
        if (e_ != cudaSuccess) return cuda_fail(e_, what); \
    } while (0)

constexpr size_t ALIGN = 256;
constexpr int64_t CHUNK = 4096;

size_t real_size(int prec) { return prec == FVLBM_FP64 ? 8 : 4; }
// bytes of stored state per cell: 9 values, or for the 16-bit split format
// 3 FP32 moments + 6 16-bit non-equilibrium values
size_t state_bytes(int prec) {
    return prec == FVLBM_FP64 ? 72 : (prec == FVLBM_FP32_DEV ? 36 : 24);
}

// Tile structure of the fused stage kernel.  Tiles are runs of consecutive
// cells (internal order), cut where tile and 1-ring (face neighbours outside
// the tile) would exceed the CTA's `tile` threads, or where the local cells
// (tile, 1-ring, 2-ring = face neighbours of the 1-ring outside tile and
// 1-ring) or the tile's boundary faces would exceed the kernel's shared-memory
// capacity.  Every slot of a tile or 1-ring cell has a link word (see
// fvlbm_internal.h): the local index of its neighbour, which direction of each
// pair leaves through it, its kind and, for tile cells, the face-table row of
// what enters.
struct TilePlan {
    int tile = 0;
    int64_t n_tiles = 0;
    std::vector<TileRec> rec;       // [n_tiles]
    std::vector<int32_t> halo;      // 1-ring then 2-ring of each tile
    std::vector<uint32_t> link;     // [n_cell][maxf] link words of the tile cells
    std::vector<uint32_t> r1link;   // [1-ring entries][maxf] link words
    int64_t n_r1 = 0;               // 1-ring entries
    int32_t max_local = 0, max_faces = 0, max_ghosts = 0;
    int64_t short_tiles = 0;        // tiles cut below the length asked for by the capacity
    int64_t sum_len = 0, sum_ring1 = 0, sum_local = 0;   // over the tiles
    // filled when the plan is verified (fvlbm_plan_info): modelled
    // shared-memory wavefronts of the warp accesses, and failed invariants
    bool verify = false;
    double face_groups = 0, face_waves = 0, gather_groups = 0, gather_waves = 0;
    int64_t violations = 0;
    std::string first_violation;
};

// Shared-memory capacity of the fused kernel for a tile size (TileDims).
// loop: in the resident loop's layout, whose face table is of fixed size.
bool tile_dims(int tile, int maxf, int rsize, bool loop, int& ls, int& ghosts, size_t& bytes) {
#define FVLBM_TD(T_)                                                                                         \
    case T_:                                                                                                 \
        ls = TileDims<T_, 4, 4>::LS;                                                                         \
        ghosts = rsize == 4 && !loop ? TileDims<T_, 4, 4>::MAX_GHOSTS : TileDims<T_, 4, 4>::GHOSTS;           \
        bytes = maxf <= 4 ? (rsize == 4 ? TileDims<T_, 4, 4>::BYTES : TileDims<T_, 4, 8>::BYTES)             \
                          : (rsize == 4 ? TileDims<T_, 8, 4>::BYTES : TileDims<T_, 8, 8>::BYTES);            \
        return true;
    switch (tile) {
        FVLBM_TD(64)
        FVLBM_TD(128)
        FVLBM_TD(256)
        FVLBM_TD(512)
        FVLBM_TD(1024)
    }
#undef FVLBM_TD
    return false;
}

struct TileScratch {
    std::vector<int64_t> stamp;
    std::vector<int32_t> loc;
    std::vector<int64_t> r1, r2;
    std::vector<uint32_t> t_link, r_link;
    int64_t gen = 0;
};

// Direction pairs (A, B) of the link words, as in fvlbm_device.cuh.
constexpr int PAIR_A[4] = {1, 2, 5, 6}, PAIR_B[4] = {3, 4, 7, 8};
constexpr int EXI[FVLBM_Q] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
constexpr int EYI[FVLBM_Q] = {0, 0, 1, 0, -1, 1, 1, -1, -1};

// Pair bits of slot k of cell i (internal numbers): bit p set when direction A
// of pair p leaves the cell through the face (e.n > 0).  A pair parallel to an
// interior face (e.n = 0, zero flux) is given to the side with the smaller
// (cell, slot), so that the two sides always hold complementary bits.
uint32_t pair_bits(const Mesh& M, int64_t i, int k) {
    const Slot& S = M.slots[(size_t)M.perm[i] * MAXP + k];
    bool first = true;
    if (S.kind == SK_INTERIOR) {
        const int64_t j = M.iperm[S.nb];
        first = i < j || (i == j && k < S.nb_slot);
    }
    uint32_t m = 0;
    for (int p = 0; p < 4; p++) {
        const bool a = (S.outmask >> (PAIR_A[p] - 1)) & 1u, b = (S.outmask >> (PAIR_B[p] - 1)) & 1u;
        if (a || (!b && first)) m |= 1u << p;
    }
    return m;
}

uint32_t link_kind(const Mesh& M, const Slot& S) {
    switch (S.kind) {
        case SK_INTERIOR: return LK_FLOW;
        case SK_WALL: return LK_WALL;
        case SK_INLET: return LK_INLET;
        case SK_OUTLET: return M.bcs[S.bc].external ? LK_OUTLET : LK_PRESSURE;
        case SK_SYMMETRY: return LK_SYMMETRY;
        default: return LK_NONE;
    }
}

uint32_t link_word(uint32_t nb, uint32_t pairs, uint32_t kind, uint32_t row) {
    return nb | pairs << LINK_PAIR_SHIFT | kind << LINK_KIND_SHIFT | row << LINK_ROW_SHIFT;
}
uint32_t word_nb(uint32_t w) { return w & LINK_NB_MASK; }
uint32_t word_pairs(uint32_t w) { return (w >> LINK_PAIR_SHIFT) & 0xFu; }
uint32_t word_kind(uint32_t w) { return (w >> LINK_KIND_SHIFT) & 7u; }
uint32_t word_row(uint32_t w) { return w >> LINK_ROW_SHIFT; }

}  // namespace

// What the planner asks of a mesh, by internal cell number: the mesh's own slots are
// some kilobyte per cell, which a plan goes over several times and a solver may have
// two plans and tries more (host time to set up a solver of 78k quads 53 ms with the
// slots, 29 with this).  Kept with the mesh.
struct fvlbm::Adjacency {
    int maxf = 0;
    std::vector<uint8_t> nf;       // [n_cell] faces
    std::vector<int32_t> nbr;      // [n_cell][maxf] neighbour, -1 at a boundary or an unused slot
    std::vector<uint32_t> word;    // [n_cell][maxf] pairs and kind where a link word has them, the
                                   // face's slot in the neighbour in place of the row
    Adjacency(const Mesh& M, int maxf_) : maxf(maxf_) {
        const int64_t n = M.n_cell;
        nf.resize((size_t)n);
        nbr.assign((size_t)n * maxf, -1);
        word.assign((size_t)n * maxf, link_word(0, 0, LK_NONE, 0));
        for (int64_t c = 0; c < n; c++) {   // in the slots' own order
            const int64_t i = M.iperm[c];
            nf[i] = (uint8_t)M.nf[c];
            for (int k = 0; k < M.nf[c]; k++) {
                const Slot& S = M.slots[(size_t)c * MAXP + k];
                const size_t w = (size_t)i * maxf + k;
                const bool inner = S.kind == SK_INTERIOR;
                if (inner) nbr[w] = (int32_t)M.iperm[S.nb];
                word[w] = link_word(0, pair_bits(M, i, k), link_kind(M, S), inner ? (uint32_t)S.nb_slot : 0u);
            }
        }
    }
    int32_t at(int64_t i, int k) const { return nbr[(size_t)i * maxf + k]; }
};

namespace {

// Link words of the tile [c0, c0 + len): local numbering tile cells, 1-ring,
// 2-ring.  False when it exceeds ls local cells or `ghosts` boundary faces, or
// when tile and 1-ring together exceed the CTA's `threads` (the kernel gives
// every thread at most one gradient to compute).
bool try_tile(const Adjacency& A, int64_t c0, int len, int threads, int ls, int ghosts, TileScratch& W,
              int& n_local, int& n_faces, int& n_ghosts) {
    const int64_t g = ++W.gen;
    const int maxf = A.maxf;
    int nl = 0;
    for (int64_t i = c0; i < c0 + len; i++) {
        W.stamp[i] = g;
        W.loc[i] = nl++;
    }
    W.r1.clear();
    W.r2.clear();
    for (int64_t i = c0; i < c0 + len; i++)
        for (int k = 0; k < A.nf[i]; k++) {
            const int64_t j = A.at(i, k);
            if (j >= 0 && W.stamp[j] != g) {
                W.stamp[j] = g;
                W.loc[j] = nl++;
                W.r1.push_back(j);
            }
        }
    const int n1 = (int)W.r1.size();
    if (nl > ls || len + n1 > threads) return false;
    for (int64_t j : W.r1)
        for (int k = 0; k < A.nf[j]; k++) {
            const int64_t q = A.at(j, k);
            if (q >= 0 && W.stamp[q] != g) {
                W.stamp[q] = g;
                W.loc[q] = nl++;
                W.r2.push_back(q);
            }
        }
    if (nl > ls) return false;
    // 1-ring and 2-ring each in global order: the kernel gathers them with
    // consecutive threads, which then share the sectors of a 32-cell block
    std::sort(W.r1.begin(), W.r1.end());
    std::sort(W.r2.begin(), W.r2.end());
    int x = len;
    for (int64_t j : W.r1) W.loc[j] = x++;
    for (int64_t q : W.r2) W.loc[q] = x++;
    W.t_link.resize((size_t)len * maxf);
    W.r_link.resize((size_t)n1 * maxf);
    int n_ghost = 0, n_slots = 0, inner = 0;
    for (int li = 0; li < len; li++) {
        const int64_t i = c0 + li;
        for (int k = 0; k < maxf; k++) {
            uint32_t& w = W.t_link[(size_t)li * maxf + k];
            if (k >= A.nf[i]) {
                w = link_word((uint32_t)li, 0, LK_NONE, 0);   // row 0: finite, read with weight zero
                continue;
            }
            const uint32_t a = A.word[(size_t)i * maxf + k];
            const int32_t j = A.at(i, k);
            n_slots++;
            if (j >= 0) {
                const uint32_t lj = (uint32_t)W.loc[j];
                inner += (int)lj < len;
                w = link_word(lj, word_pairs(a), LK_FLOW, word_row(a) * threads + lj);
            } else {
                if (n_ghost == ghosts) return false;
                w = link_word((uint32_t)li, word_pairs(a), word_kind(a), (uint32_t)(maxf * threads + n_ghost++));
            }
        }
    }
    for (int e = 0; e < n1; e++) {
        const int64_t i = W.r1[e];
        for (int k = 0; k < maxf; k++) {
            uint32_t& w = W.r_link[(size_t)e * maxf + k];
            const uint32_t a = A.word[(size_t)i * maxf + k];
            const int32_t q = k < A.nf[i] ? A.at(i, k) : -1;
            if (q >= 0) {
                const uint32_t lq = (uint32_t)W.loc[q];
                w = link_word(lq, word_pairs(a), (int)lq < len ? LK_FLOW : LK_OTHER, 0);
            } else {
                w = link_word((uint32_t)(len + e), word_pairs(a), word_kind(a), 0);   // boundary or unused slot
            }
        }
    }
    n_local = nl;
    n_faces = n_slots - inner / 2;
    n_ghosts = n_ghost;
    return true;
}

// Shared-memory wavefronts of a warp's 16-byte accesses relative to the four
// that a conflict-free one takes: eight lanes at a time, eight 16-byte banks;
// a group takes as many as the most distinct rows that share a bank.
double bank_waves(const int* idx, int n) {
    double m = 0;
    for (int b = 0; b < n; b += 8) {
        int v[8], cnt[8] = {0}, w = 0;
        const int e = std::min(8, n - b);
        for (int q = 0; q < e; q++) v[q] = idx[b + q];
        std::sort(v, v + e);
        for (int q = 0; q < e; q++)
            if (q == 0 || v[q] != v[q - 1]) w = std::max(w, ++cnt[v[q] & 7]);
        m += w;
    }
    return m / ((n + 7) / 8);
}

// Checks of one tile's plan (fvlbm_plan_info), against the mesh: every slot
// links to its neighbour's local index (boundary and unused slots to the cell
// itself, unused slots to row 0), what enters through an interior face is read
// from the row that the neighbour writes there, no two boundary faces share a
// ghost row, each (face, direction) between local cells has exactly one writer,
// and tile + 1-ring and the local cells fit the CTA; then the modelled
// wavefronts of the face-table accesses (a slot's own row, written and read
// without conflict, and the neighbour's row) and of the neighbour gathers.
void verify_tile(const Mesh& M, int maxf, int64_t c0, int len, int threads, int ls, int ghosts, int nl,
                 const TileScratch& W, TilePlan& P) {
    auto bad = [&](const char* what, int64_t cell) {
        if (P.violations++ == 0) {
            char b[200];
            std::snprintf(b, sizeof b, "tile at cell %lld: %s (cell %lld)", (long long)c0, what, (long long)cell);
            P.first_violation = b;
        }
    };
    const int n1 = (int)W.r1.size();
    if (len + n1 > threads) bad("tile and 1-ring exceed the CTA's threads", c0);
    if (nl > ls) bad("local cells exceed the shared-memory capacity", c0);
    std::vector<char> taken((size_t)ghosts, 0);
    for (int li = 0; li < len + n1; li++) {
        const int64_t i = li < len ? c0 + li : W.r1[li - len];
        const int64_t c = M.perm[i];
        for (int k = 0; k < maxf; k++) {
            const uint32_t w = li < len ? W.t_link[(size_t)li * maxf + k] : W.r_link[(size_t)(li - len) * maxf + k];
            if (k >= M.nf[c]) {
                if (word_kind(w) != LK_NONE || word_nb(w) != (uint32_t)li || word_row(w) != 0)
                    bad("unused slot not linked to itself and row 0", i);
                continue;
            }
            const Slot& S = M.slots[(size_t)c * MAXP + k];
            for (int p = 0; p < 4; p++) {
                // the direction given to this side must not enter through the face
                const int a = (word_pairs(w) >> p) & 1u ? PAIR_A[p] : PAIR_B[p];
                if (EXI[a] * S.nx + EYI[a] * S.ny < 0) bad("a direction that enters marked as leaving", i);
            }
            if (S.kind != SK_INTERIOR) {
                if (word_nb(w) != (uint32_t)li) bad("boundary slot not linked to itself", i);
                if (word_kind(w) != link_kind(M, S)) bad("boundary slot of the wrong kind", i);
                if (li >= len) continue;
                const int64_t row = (int64_t)word_row(w) - (int64_t)maxf * threads;
                if (row < 0 || row >= ghosts) bad("ghost row outside the face table", i);
                else if (taken[row]++) bad("two boundary faces share a ghost row", i);
                continue;
            }
            const int64_t j = M.iperm[S.nb];
            const int lj = W.loc[j];
            if (word_nb(w) != (uint32_t)lj) bad("slot not linked to its neighbour", i);
            if (li >= len) {
                if (word_kind(w) != (lj < len ? LK_FLOW : LK_OTHER)) bad("a 1-ring face wrongly marked", i);
                continue;
            }
            if (word_kind(w) != LK_FLOW) bad("interior slot of the wrong kind", i);
            if (lj >= len + n1) {
                bad("a tile cell's neighbour is not in the tile or its 1-ring", i);
                continue;
            }
            if (word_row(w) != (uint32_t)(S.nb_slot * threads + lj)) bad("a face not read from the row its neighbour writes", i);
            const uint32_t wj = lj < len ? W.t_link[(size_t)lj * maxf + S.nb_slot]
                                         : W.r_link[(size_t)(lj - len) * maxf + S.nb_slot];
            if (word_kind(wj) != LK_FLOW || word_nb(wj) != (uint32_t)li) bad("the two sides of a face do not link to each other", i);
            if ((word_pairs(w) ^ word_pairs(wj)) != 0xFu) bad("a (face, direction) without exactly one writer", i);
        }
    }
    // modelled wavefronts of the warp accesses through one slot (used slots only)
    int idx[BLK];
    for (int w = 0; w * BLK < len; w++)
        for (int k = 0; k < maxf; k++) {
            int n = 0;
            bool used = k < 3;
            for (int li = w * BLK; li < std::min(len, (w + 1) * BLK); li++) {
                idx[n++] = (int)word_row(W.t_link[(size_t)li * maxf + k]);
                used |= k < M.nf[M.perm[c0 + li]];
            }
            if (!used) continue;
            P.face_groups += 3;
            P.face_waves += 2 + bank_waves(idx, n);
        }
    for (int w = 0; w * BLK < len + n1; w++)
        for (int k = 0; k < maxf; k++) {
            int n = 0;
            bool used = k < 3;
            for (int l = w * BLK; l < std::min(len + n1, (w + 1) * BLK); l++) {
                const int64_t c = l < len ? c0 + l : W.r1[l - len];
                idx[n++] = (int)word_nb(l < len ? W.t_link[(size_t)l * maxf + k] : W.r_link[(size_t)(l - len) * maxf + k]);
                used |= k < M.nf[M.perm[c]];
            }
            if (!used) continue;
            P.gather_groups += 1;
            P.gather_waves += bank_waves(idx, n);
        }
}

// max_len: most cells of a tile (0: as many as fit).  max_tiles: most tiles (0: any
// number); FVLBM_ERR_UNSUPPORTED as soon as more are sure to be needed.
// loop: for the resident loop.
int make_tiles(const Mesh& M, const Adjacency& A, int tile, int rsize, bool loop, TilePlan& P, bool verify,
               int max_len = 0, int64_t max_tiles = 0) {
    int ls = 0, ghosts = 0;
    size_t bytes = 0;
    const int maxf = A.maxf;
    if (!tile_dims(tile, maxf, rsize, loop, ls, ghosts, bytes)) return fail(FVLBM_ERR_ARG, "unsupported tile size %d", tile);
    const int64_t n = M.n_cell;
    P = TilePlan{};
    P.tile = tile;
    P.verify = verify;
    P.link.assign((size_t)n * maxf, 0);
    TileScratch W;
    W.stamp.assign(n, 0);
    W.loc.assign(n, 0);
    // tiles cover the owned cells; ghost cells of a partition only appear in halos
    const int64_t n_own = M.n_owned;
    int64_t c0 = 0;
    int32_t inst = 0;
    if (max_len <= 0 || max_len > tile) max_len = tile;
    int guess = max_len;   // neighbouring tiles have similar lengths: start one block above the last
    while (c0 < n_own) {
        int len = (int)std::min<int64_t>(guess, n_own - c0);
        int nl = 0, nf = 0, ng = 0;
        while (!try_tile(A, c0, len, tile, ls, ghosts, W, nl, nf, ng)) {
            if (len == 1)
                return fail(FVLBM_ERR_UNSUPPORTED, "cell %lld: its halo exceeds the fused stage's capacity",
                            (long long)c0);
            len = len > BLK ? (len - 1) / BLK * BLK : len / 2;
        }
        guess = std::min(max_len, (len + BLK) / BLK * BLK);
        if (len < std::min<int64_t>(max_len, n_own - c0)) P.short_tiles++;
        P.sum_len += len;
        P.sum_ring1 += (int64_t)W.r1.size();
        P.sum_local += nl;
        if (verify) verify_tile(M, maxf, c0, len, tile, ls, ghosts, nl, W, P);
        std::copy(W.t_link.begin(), W.t_link.end(), P.link.begin() + (size_t)c0 * maxf);
        // instances are contiguous in the internal order, and a face never joins two
        while (inst + 1 < M.n_inst && c0 >= M.inst_begin[inst + 1]) inst++;
        TileRec R{};
        R.c0 = (int32_t)c0;
        R.nt = len;
        R.h0 = (int32_t)P.halo.size();
        R.nh = (int32_t)(W.r1.size() + W.r2.size());
        R.q0 = (int32_t)P.n_r1;
        R.n1 = (int32_t)W.r1.size();
        R.inst = M.n_inst == 1 || c0 + len <= M.inst_begin[inst + 1] ? inst : -1;
        P.rec.push_back(R);
        for (int64_t j : W.r1) P.halo.push_back((int32_t)j);
        for (int64_t q : W.r2) P.halo.push_back((int32_t)q);
        if (P.halo.size() >= (size_t)1 << 31)
            return fail(FVLBM_ERR_UNSUPPORTED, "fused stage: the halos exceed its 32-bit indexing; use kernel = 1");
        P.r1link.insert(P.r1link.end(), W.r_link.begin(), W.r_link.end());
        P.n_r1 += R.n1;
        c0 += len;
        if (max_tiles > 0 && (int64_t)P.rec.size() + (n_own - c0 + max_len - 1) / max_len > max_tiles)
            return fail(FVLBM_ERR_UNSUPPORTED, "more than %lld tiles", (long long)max_tiles);
        P.max_ghosts = std::max(P.max_ghosts, ng);
        P.max_local = std::max(P.max_local, nl);
        P.max_faces = std::max(P.max_faces, nf);
    }
    P.n_tiles = (int64_t)P.rec.size();
    return FVLBM_OK;
}

// Offsets of every array inside the workspace (0 size when a strategy does not use it).
struct Layout {
    int64_t np, n_chunk;
    int maxf;
    int strategy;
    int block;
    bool pingpong;   // single-stage scheme on the fused stage: the state alternates between fa and fb
    TilePlan tp;
    int64_t n_ghost;   // two-kernel stage: boundary slots of owned cells (ghost records)
    size_t off_link, off_geo, off_bctag, off_nbr, off_area, off_grp, off_inst, off_bc, off_fa, off_fb, off_fc, off_rprev,
        off_fv, off_uold, off_part, off_red, off_conv, off_chunk, off_flag, off_tiles, off_halo,
        off_r1link, off_iperm, total;
    // resident stage loop (small solvers)
    TilePlan rp;
    bool resident;
    const TilePlan& res_plan() const { return rp.n_tiles > 0 ? rp : tp; }   // tp when it serves both
    size_t off_rlink, off_rtiles, off_rhalo, off_rr1link, off_xchg;
};

constexpr size_t SMEM_LIMIT = 227 * 1024;
// shortest tiles (FP32: 16 / 32 / 48 / 96 cells 2.06 / 1.56 / 1.61 / 1.71 us per stage of 2,048
// triangles, 2.28 / 2.17 / 1.96 / 1.85 of 3,600 quads; FP64: 4 / 8 / 16 cells 6.2 / 5.5 / 5.4 of 512)
constexpr int RES_MIN_CELLS(int rsize) { return rsize == 4 ? 48 : 16; }

// Streaming multiprocessors of a device (152 on GB300 when no device answers).
int device_sms(int device) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || n <= 0) {
        cudaGetLastError();
        n = 152;
    }
    return n;
}
constexpr int64_t PLANE_ALIGN = 1024;  // cell arrays hold whole blocks and whole tiles of the largest size

int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// What the resident loop's exchange relies on besides: who reads from a tile is read
// by it (so that a tile that has its neighbours' cells of a stage knows that they
// have read its older ones).
void verify_exchange(TilePlan& P) {
    int64_t n = 0;
    for (const TileRec& R : P.rec) n = std::max<int64_t>(n, R.c0 + R.nt);
    std::vector<int32_t> owner((size_t)n);
    for (size_t t = 0; t < P.rec.size(); t++)
        std::fill_n(owner.begin() + P.rec[t].c0, P.rec[t].nt, (int32_t)t);
    std::vector<std::pair<int32_t, int32_t>> reads;
    for (size_t t = 0; t < P.rec.size(); t++)
        for (int32_t h = 0; h < P.rec[t].nh; h++) reads.emplace_back((int32_t)t, owner[P.halo[P.rec[t].h0 + h]]);
    std::sort(reads.begin(), reads.end());
    reads.erase(std::unique(reads.begin(), reads.end()), reads.end());
    for (const auto& r : reads)
        if (!std::binary_search(reads.begin(), reads.end(), std::make_pair(r.second, r.first)) && P.violations++ == 0)
            P.first_violation = "a tile reads from one that does not read from it";
}

// The resident stage loop's plan (fvlbm_resident.cuh), if the solver is small
// enough: one tile per SM, as long as the SM's share of the cells but not below
// a length at which the halo outgrows the tile; in FP32 also two to four of the
// largest tiles per SM.  The limits are what fits on the GPU at once, below which it
// was the faster way throughout (us per FP32 stage, here / streaming: 40k cells 3.1 /
// 4.9, 68k 3.8 / 5.6, 78k 5.6 / 6.5, 90k 5.9 / 6.4; FP64 3.6k cells 6.6, streaming 10k
// cells 17.5).
// adjacency(): the mesh's, formed when the first plan is tried.
template <typename Get> int make_resident(const Mesh& M, int maxf, Get adjacency, int rsize, int sms, TilePlan& P, bool verify) {
    const int64_t n = M.n_owned;
    const int most = rsize == 8 ? RES_TILE_FP64 : RES_TILE;
    P = TilePlan{};
    for (int ctas = 1; ctas <= resident_ctas(rsize, maxf); ctas++) {
        const int64_t share = std::max<int64_t>((n + ctas * sms - 1) / (ctas * sms), RES_MIN_CELLS(rsize));
        for (int tile = ctas > 1 ? most : rsize == 8 ? RES_TILE_FP64 : RES_TILE / 2; tile <= most; tile *= 2) {
            // a compact tile of q cells has about 4.3 sqrt(q) 1-ring cells
            if (share + 4.3 * std::sqrt((double)share) > tile) continue;
            // equal tiles; where a few are cut shorter and there are too many, as long as they fit
            for (int64_t len : {std::min<int64_t>(share, tile), (int64_t)tile}) {
                if (len == tile && ctas < std::min(3, resident_ctas(rsize, maxf))) continue;
                int rc = make_tiles(M, adjacency(), tile, rsize, true, P, verify, (int)len, (int64_t)ctas * sms);
                if (rc == FVLBM_OK) {
                    if (verify) verify_exchange(P);
                    return FVLBM_OK;
                }
                P = TilePlan{};
                if (rc != FVLBM_ERR_UNSUPPORTED) return rc;
                clear_error();
            }
        }
    }
    return FVLBM_OK;   // none: P.n_tiles == 0
}

// kernel: 1 two-kernel, 128/256/512/1024 fused with that tile size, 0
// automatic.  The automatic choice, from measurements on GB300:
//  - FP32 / 16-bit: 512-thread tiles once the mesh gives every SM a tile of
//    512 (the fastest on large batches), 256-thread tiles down to a quarter of
//    the SMs' worth of them (e.g. the 128^2 cavity, the 60k-cell cylinder),
//    128-thread tiles below: a fused stage launches one kernel per stage where
//    the two-kernel stage launches two, which is what small meshes wait on;
//  - FP64: the two-kernel stage (it spends fewer FP64 operations: no 1-ring
//    gradients, and the FP64 mode is bound by GB300's FP64 units) except on
//    meshes of fewer than 32 cells per SM: fused 128, one launch per stage.  (With four
//    lanes per cell two kernels are faster there as well, 11.0 us per stage of 512 cells
//    against 16.6; such meshes run in the resident loop, 5.5, but for single stages.)
// The two-kernel stage shrinks its blocks (down to 32 threads) so that small
// meshes still spread over the SMs.
// loop: false leaves the resident loop and its arrays out.
int make_layout(const fvlbm_mesh& mesh, int prec, int scheme, int kernel, Layout& L, int sms, bool verify = false,
                bool loop = true) {
    const Mesh& M = mesh.m;
    L = Layout{};
    L.np = round_up(M.n_cell, PLANE_ALIGN);
    L.maxf = M.max_faces <= 4 ? 4 : 8;
    L.n_chunk = 0;
    for (int k = 0; k < M.n_inst; k++) L.n_chunk += (M.inst_begin[k + 1] - M.inst_begin[k] + CHUNK - 1) / CHUNK;
    const size_t R = real_size(prec), S = state_bytes(prec);
    if (kernel != 0 && kernel != 1 && kernel != 128 && kernel != 256 && kernel != 512 && kernel != 1024)
        return fail(FVLBM_ERR_ARG, "params.kernel = %d: use 0, 1, 128, 256, 512 or 1024", kernel);
    int tile = kernel;
    if (kernel == 0) {
        const int64_t n = M.n_owned;
        auto fits = [&](int t) {
            int ls = 0, fs = 0;
            size_t smem = 0;
            tile_dims(t, L.maxf, (int)R, false, ls, fs, smem);
            return smem <= SMEM_LIMIT;
        };
        if (prec == FVLBM_FP64) tile = n < 32 * (int64_t)sms ? 128 : 1;
        else if (n >= 512 * (int64_t)sms && fits(512)) tile = 512;
        else if (n >= 64 * (int64_t)sms) tile = 256;
        else tile = 128;
    }
    L.strategy = tile == 0 || tile == 1 ? STRATEGY_TWO_KERNEL : STRATEGY_TILE;
    auto adjacency = [&]() -> const Adjacency& {
        std::lock_guard<std::mutex> lock(mesh.plan_mutex);
        if (!mesh.adjacency) mesh.adjacency = std::make_shared<const Adjacency>(M, L.maxf);
        return *mesh.adjacency;
    };
    // the resident loop: chosen with the automatic kernel only; parts of a
    // partitioned mesh exchange after every stage and never use it
    L.resident = false;
    if (loop && kernel == 0 && M.n_owned == M.n_cell && M.n_owned > 0) {
        int rc = make_resident(M, L.maxf, adjacency, (int)R, sms, L.rp, verify);
        if (rc) return rc;
        L.resident = L.rp.n_tiles > 0;
    }
    // FP64: small blocks, whose warps the SMs' quarters share more evenly (250k-cell
    // cavity 130 us per stage with 64 threads, 134 with 256)
    L.block = prec == FVLBM_FP64 ? 64 : 256;
    while (prec != FVLBM_FP64 && L.block > 32 && (M.n_owned + L.block - 1) / L.block < 2 * sms) L.block /= 2;
    if (L.strategy == STRATEGY_TILE) {
        int ls = 0, fs = 0;
        size_t smem = 0;
        tile_dims(tile, L.maxf, (int)R, false, ls, fs, smem);
        if (smem > SMEM_LIMIT)
            return fail(FVLBM_ERR_UNSUPPORTED, "fused stage with %d-cell tiles needs %zu B of shared memory (limit %zu)",
                        tile, smem, SMEM_LIMIT);
        // the resident loop's tiles, where they are of this size and nearly full (a tile of q
        // cells has about 4.3 sqrt(q) 1-ring cells), serve both.  Shorter ones would make
        // the stage kernels compute more of their halo: eight solvers of the 30k-cell hybrid
        // side by side 12.9 us per FP32 stage of all with tiles of 99 cells, 9.0 with 180
        const double root = 0.5 * (std::sqrt(4.3 * 4.3 + 4.0 * tile) - 4.3), full = root * root;
        int rc = FVLBM_OK;
        if (L.resident && L.rp.tile == tile && L.rp.sum_len >= 0.85 * full * L.rp.n_tiles) std::swap(L.tp, L.rp);
        else rc = make_tiles(M, adjacency(), tile, (int)R, false, L.tp, verify);
        if (rc) return rc;
        // the fused kernel indexes its blocked arrays in 32 bits
        const uint64_t lim = (uint64_t)1 << 32;
        if ((uint64_t)L.np * 3 * L.maxf >= lim || (uint64_t)L.tp.n_r1 * L.maxf >= lim)
            return fail(FVLBM_ERR_UNSUPPORTED, "fused stage: %lld cells exceed its 32-bit indexing; use kernel = 1",
                        (long long)M.n_cell);
    }
    const bool tiled = L.strategy == STRATEGY_TILE, two = !tiled;
    L.pingpong = tiled && (scheme == FVLBM_EULER || scheme == FVLBM_AB2);
    size_t o = 0;
    auto take = [&](size_t bytes) {
        size_t r = o;
        o += (bytes + ALIGN - 1) / ALIGN * ALIGN;
        return r;
    };
    const size_t plane = (size_t)L.np, slots = plane * L.maxf;
    L.n_ghost = two ? M.n_bface : 0;
    L.off_link = take(4 * slots);
    L.off_geo = take(2 * R * 3 * slots);
    L.off_bctag = take(2 * slots);
    L.off_nbr = take(two ? 4 * slots : 0);
    L.off_area = take(8 * plane);
    L.off_grp = take(4 * plane);
    L.off_iperm = take(4 * plane);
    L.off_inst = take(sizeof(InstParam) * M.n_inst);
    L.off_bc = take(sizeof(BcParam) * std::max<size_t>(1, M.bcs.size()));
    L.off_tiles = take(tiled ? sizeof(TileRec) * (size_t)L.tp.n_tiles : 0);
    L.off_halo = take(tiled ? 4 * L.tp.halo.size() : 0);
    L.off_r1link = take(tiled ? 4 * (size_t)L.tp.n_r1 * L.maxf : 0);
    const bool own_plan = L.rp.n_tiles > 0;
    L.off_rlink = own_plan ? take(4 * slots) : L.off_link;
    L.off_rtiles = own_plan ? take(sizeof(TileRec) * (size_t)L.rp.n_tiles) : L.off_tiles;
    L.off_rhalo = own_plan ? take(4 * L.rp.halo.size()) : L.off_halo;
    L.off_rr1link = own_plan ? take(4 * (size_t)L.rp.n_r1 * L.maxf) : L.off_r1link;
    L.off_fa = take(S * plane);   // everything before this is uploaded once
    L.off_fb = (scheme == FVLBM_RK2 || scheme == FVLBM_RK4 || L.pingpong) ? take(S * plane) : 0;
    L.off_xchg = take(L.resident ? 2 * 16 * (size_t)resident_units(S) * plane : 0);
    L.off_fc = (scheme == FVLBM_RK4 && tiled) ? take(S * plane) : 0;
    L.off_rprev = scheme == FVLBM_AB2 ? take(R * plane * FVLBM_Q) : 0;
    L.off_fv = take(two ? 4 * R * (slots + (size_t)L.n_ghost) : 0);
    L.off_uold = take(16 * plane);
    L.off_part = take(16 * RED_PARTS * (size_t)std::max<int64_t>(1, L.n_chunk));
    L.off_red = take(16 * (size_t)M.n_inst);
    L.off_conv = take(8 * plane * FVLBM_Q);
    L.off_chunk = take(24 * (size_t)std::max<int64_t>(1, L.n_chunk) + 8 * (size_t)(M.n_inst + 1));
    L.off_flag = take(16);
    L.total = o;
    return FVLBM_OK;
}

int check_params(const Mesh& M, const fvlbm_params* params, int32_t n_params) {
    if (M.n_cell >= ((int64_t)1 << 31)) return fail(FVLBM_ERR_ARG, "more than 2^31 - 1 cells");
    if (!params || !(n_params == 1 || n_params == M.n_inst))
        return fail(FVLBM_ERR_ARG, "params: need 1 or %d entries, got %d", M.n_inst, n_params);
    for (int32_t k = 0; k < n_params; k++) {
        const fvlbm_params& p = params[k];
        if (!(p.tau > 0) || !(p.dt >= 0) || !(p.cfl >= 0) || !(p.u_max >= 0) || !(p.rho0 > 0))
            return fail(FVLBM_ERR_ARG, "params[%d]: tau, rho0 must be > 0; dt, cfl, u_max >= 0", k);
        if (p.scheme < FVLBM_EULER || p.scheme > FVLBM_RK4) return fail(FVLBM_ERR_ARG, "params[%d]: bad scheme", k);
        if (p.precision < FVLBM_FP64 || p.precision > FVLBM_BF16_DEV)
            return fail(FVLBM_ERR_ARG, "params[%d]: bad precision", k);
        if (p.scheme != params[0].scheme || p.precision != params[0].precision || p.device != params[0].device ||
            p.kernel != params[0].kernel)
            return fail(FVLBM_ERR_ARG, "params[%d]: scheme, precision, device and kernel must match params[0]", k);
    }
    if (M.bcs.size() >= 65536) return fail(FVLBM_ERR_ARG, "too many boundary tags (%zu)", M.bcs.size());
    return FVLBM_OK;
}

// Largest speed the instance is set up with: |U|_max of Eq. (CFL) when not given.
double instance_umax(const Mesh& M, int k, const fvlbm_params& p) {
    if (p.u_max > 0) return p.u_max;
    double u = std::hypot(p.u0[0], p.u0[1]);
    for (int32_t b = M.inst_bc_begin[k]; b < M.inst_bc_begin[k + 1]; b++) {
        const fvlbm_bc& c = M.bcs[b];
        if (c.kind == FVLBM_BC_WALL) u = std::max(u, std::hypot(c.u_w[0], c.u_w[1]));
        if (c.kind == FVLBM_BC_INLET || c.kind == FVLBM_BC_OUTLET) u = std::max(u, std::hypot(c.u_inf[0], c.u_inf[1]));
    }
    return u;
}

// Index of component c of cell i in a blocked array of ncomp components.
inline size_t blk(int64_t i, int c, int ncomp) {
    return (size_t)((i >> BLK_SHIFT) * ((int64_t)ncomp << BLK_SHIFT) + ((int64_t)c << BLK_SHIFT) + (i & (BLK - 1)));
}

template <typename T>
void pack_geometry(const Mesh& M, const Layout& L, std::vector<unsigned char>& host) {
    const int64_t n = M.n_cell;
    const int maxf = L.maxf;
    const bool two = L.strategy == STRATEGY_TWO_KERNEL;
    unsigned char* H = host.data();
    uint32_t* link = (uint32_t*)(H + L.off_link);   // units of four words
    T* geo = (T*)(H + L.off_geo);                   // 16-byte units of 2-vectors (GeoRef)
    uint16_t* bctag = (uint16_t*)(H + L.off_bctag);
    double* area = (double*)(H + L.off_area);
    int32_t* grp = (int32_t*)(H + L.off_grp);
    int32_t* iperm = (int32_t*)(H + L.off_iperm);
    for (int64_t c = 0; c < n; c++) iperm[c] = (int32_t)M.iperm[c];
    int32_t* nbr = two ? (int32_t*)(H + L.off_nbr) : nullptr;
    constexpr int PER = 16 / (2 * sizeof(T));   // 2-vectors per unit
    const int units = maxf / PER;
    // word of slot k, and 2-vector v of slot k
    auto word = [&](int64_t i, int k) { return 4 * blk(i, k / 4, maxf / 4) + k % 4; };
    auto vec = [&](int64_t i, int v, int k) { return geo + 2 * (PER * blk(i, v * units + k / PER, 3 * units) + k % PER); };
    int64_t next = 0;
    int32_t g = 0;
    for (int64_t i = 0; i < n; i++) {
        const int64_t c = M.perm[i];
        while (g + 1 < M.n_inst && c >= M.inst_begin[g + 1]) g++;
        grp[i] = g;
        area[i] = M.area[c];
        // this cell's words and vectors: word k at word(i, k), 2-vector v of slot k at vec(i, v, k)
        const size_t w0 = word(i, 0);
        T* const g0 = vec(i, 0, 0);
        const double area_i = M.area[c], cx = M.cx[c], cy = M.cy[c];
        for (int k = 0; k < maxf; k++) {
            const size_t w = w0 + (size_t)(k / 4) * 4 * BLK + k % 4;
            if (k >= M.nf[c]) {
                link[w] = two ? link_word(0, 0, LK_NONE, 0) : L.tp.link[(size_t)i * maxf + k];
                if (two) nbr[w] = (int32_t)i;
                continue;
            }
            const Slot& S = M.slots[(size_t)c * MAXP + k];
            bctag[(size_t)i * maxf + k] = (uint16_t)(S.bc < 0 ? 0 : S.bc);
            if (two) {
                const bool inner = S.kind == SK_INTERIOR;
                link[w] = link_word(0, pair_bits(M, i, k), link_kind(M, S), inner ? (uint32_t)S.nb_slot : 0u);
                nbr[w] = inner ? (int32_t)M.iperm[S.nb] : i < M.n_owned ? (int32_t)next++ : 0;
            } else {
                link[w] = L.tp.link[(size_t)i * maxf + k];
            }
            T* q = g0 + 2 * ((size_t)(k / PER) * PER * BLK + k % PER);
            const size_t next_vec = (size_t)2 * PER * BLK * units;
            q[0] = (T)S.cgx;
            q[1] = (T)S.cgy;
            q += next_vec;
            q[0] = (T)(S.px - cx);
            q[1] = (T)(S.py - cy);
            q += next_vec;
            q[0] = (T)(S.nx / area_i);
            q[1] = (T)(S.ny / area_i);
        }
    }
    // 1-ring entries: unit by unit, entry by entry
    auto pack_ring = [&](const TilePlan& P, size_t off) {
        uint32_t* r1 = (uint32_t*)(H + off);
        for (int64_t e = 0; e < P.n_r1; e++)
            for (int k = 0; k < maxf; k++) r1[4 * ((k / 4) * P.n_r1 + e) + k % 4] = P.r1link[(size_t)e * maxf + k];
    };
    if (!two) {
        pack_ring(L.tp, L.off_r1link);
        std::memcpy(H + L.off_tiles, L.tp.rec.data(), sizeof(TileRec) * L.tp.rec.size());
        std::memcpy(H + L.off_halo, L.tp.halo.data(), 4 * L.tp.halo.size());
    }
    if (L.rp.n_tiles > 0) {
        pack_ring(L.rp, L.off_rr1link);
        std::memcpy(H + L.off_rtiles, L.rp.rec.data(), sizeof(TileRec) * L.rp.rec.size());
        std::memcpy(H + L.off_rhalo, L.rp.halo.data(), 4 * L.rp.halo.size());
        uint32_t* rlink = (uint32_t*)(H + L.off_rlink);
        for (int64_t i = 0; i < n; i++)
            for (int k = 0; k < maxf; k++) rlink[word(i, k)] = L.rp.link[(size_t)i * maxf + k];
    }
}

}  // namespace

namespace fvlbm {
int workspace_bytes(const fvlbm_mesh* mesh, const fvlbm_params* params, int32_t n_params, bool loop, size_t* bytes) {
    int rc = check_params(mesh->m, params, n_params);
    if (rc) return rc;
    Layout L;
    try {
        rc = make_layout(*mesh, params[0].precision, params[0].scheme, params[0].kernel, L, device_sms(params[0].device),
                         false, loop);
    } catch (const std::bad_alloc&) {
        return fail(FVLBM_ERR_OOM, "fvlbm_workspace_bytes: out of host memory");
    }
    if (rc) return rc;
    *bytes = L.total;
    return FVLBM_OK;
}
}  // namespace fvlbm

extern "C" int fvlbm_workspace_bytes(const fvlbm_mesh* mesh, const fvlbm_params* params, int32_t n_params,
                                     size_t* bytes) {
    clear_error();
    if (!mesh || !bytes) return fail(FVLBM_ERR_ARG, "fvlbm_workspace_bytes: null argument");
    return workspace_bytes(mesh, params, n_params, true, bytes);
}

// The plans fvlbm_init would build, checked: of the stage kernels (resident: of
// the resident loop, stage_kernel = 0 when there is none).
static int plan_report(const char* what, const fvlbm_mesh* mesh, const fvlbm_params* params, int32_t n_params,
                       fvlbm_plan_info_t* info, bool resident) {
    clear_error();
    if (!mesh || !info) return fail(FVLBM_ERR_ARG, "%s: null argument", what);
    int rc = check_params(mesh->m, params, n_params);
    if (rc) return rc;
    Layout L;
    try {
        rc = make_layout(*mesh, params[0].precision, params[0].scheme, params[0].kernel, L,
                         device_sms(params[0].device), true);
    } catch (const std::bad_alloc&) {
        return fail(FVLBM_ERR_OOM, "%s: out of host memory", what);
    }
    if (rc) return rc;
    const bool tiled = resident ? L.resident : L.strategy == STRATEGY_TILE;
    const TilePlan& P = resident && L.resident ? L.res_plan() : L.tp;
    fvlbm_plan_info_t o{};
    o.stage_kernel = tiled ? P.tile : resident ? 0 : 1;
    o.slots = L.maxf;
    if (tiled && P.n_tiles > 0) {
        o.n_tiles = P.n_tiles;
        o.short_tiles = P.short_tiles;
        o.max_local_cells = P.max_local;
        o.max_faces = P.max_faces;
        o.mean_tile_cells = (double)P.sum_len / P.n_tiles;
        o.mean_ring1_cells = (double)P.sum_ring1 / P.n_tiles;
        o.mean_local_cells = (double)P.sum_local / P.n_tiles;
        o.face_table_waves = P.face_groups > 0 ? P.face_waves / P.face_groups : 0;
        o.gather_waves = P.gather_groups > 0 ? P.gather_waves / P.gather_groups : 0;
    }
    // every plan that the solver would run counts, whichever is reported
    o.violations = L.tp.violations + L.rp.violations;
    *info = o;
    if (o.violations)
        fail(FVLBM_OK, "%lld failed plan checks; first: %s", (long long)o.violations,
             (L.tp.violations ? L.tp : L.rp).first_violation.c_str());
    return FVLBM_OK;
}

extern "C" int fvlbm_plan_info(const fvlbm_mesh* mesh, const fvlbm_params* params, int32_t n_params,
                               fvlbm_plan_info_t* info) {
    return plan_report("fvlbm_plan_info", mesh, params, n_params, info, false);
}

extern "C" int fvlbm_resident_plan(const fvlbm_mesh* mesh, const fvlbm_params* params, int32_t n_params,
                                   fvlbm_plan_info_t* info) {
    return plan_report("fvlbm_resident_plan", mesh, params, n_params, info, true);
}

// What a stage costs (StageCost), from measurements of 1 to 16 solvers on streams of their
// own, us per stage of all of them, in turns / overlapping:
//   16k quads FP32    1: 2.0 / 4.8   2: 4.0 / 5.3   3: 6.0 / 5.6   4: 7.9 / 5.9   8: 15.8 / 7.0
//   30k hybrid        1: 3.0 / 5.4   2: 6.0 / 5.9   3: 9.1 / 6.4   4: 12.0 / 6.6  8: 23.9 / 9.0
//   60k hybrid        1: 3.3 / 5.8   2: 6.7 / 6.7   3: 9.9 / 7.3   4: 13.3 / 8.5
//   12k polygons      1: 2.5 / 6.9   3: 7.3 / 8.0   4: 9.7 / 8.3   8: 19.2 / 9.6
//   4k quads FP64     1: 7.0 / 18.6  3: 21.0 / 23.4 4: 28.0 / 25.3 8: 55.9 / 34.4
//   2k triangles FP32 1: 1.6 / 3.9   4: 1.8 / 4.5   8: 1.9 / 4.8   16: 3.6 / 9.2 (their launches fit side by side)
static StageCost stage_cost(const DevView& v, int prec, const ResView* r, int max_ctas) {
    StageCost c;
    const bool fp64 = prec == FVLBM_FP64, half = prec == FVLBM_FP16_DEV || prec == FVLBM_BF16_DEV, wide = v.maxf > 4;
    c.base = fp64 ? 17 : wide ? 6.5 : half ? 5.4 : 4.6;
    c.flow = v.n_cell * (fp64 ? 5.5e-4 : wide ? 3e-5 : 1.9e-5);
    if (r) {
        const int per_sm = (r->n_tiles + v.sms - 1) / v.sms;
        const double t = fp64 ? 7.0 : (per_sm == 1 ? 2.0 : per_sm <= 3 ? 3.2 : 6.0) + (wide ? 0.5 : 0.0);
        c.alone = t * (half ? 1.2 : 1.0);
        c.turn = c.alone / (max_ctas / r->n_tiles);   // so many fit side by side
        c.resident = true;
    }
    return c;
}

// The solvers of the process that have a resident loop.  Its launches are faster than
// stage kernels for one solver, but those that do not fit on the GPU together take
// turns, and three solvers that fill it are then slower than with stage kernels, which
// overlap.  So a long call looks who else steps: solvers on other streams whose last
// long call is not expected to be done yet, and, when its own last one was joined by others,
// whoever has stepped since (a program that steps several solvers in rounds and waits for
// all has none at work when a round begins).  Expected, by the host's clock and the costs
// above: events would be exact, but recording one takes 2% of a call of 100 steps.  Stage kernels need graphs, so it turns to them
// once the turns have cost as much more as those take.  The states are the same either way.
struct Crowd {
    std::mutex m;
    std::vector<fvlbm_solver*> members;
    uint64_t calls = 0;
};
static Crowd& crowd() {
    alignas(Crowd) static unsigned char place[sizeof(Crowd)];
    static Crowd* c = new (place) Crowd;   // outlives every solver
    return *c;
}
static int crowd_join(fvlbm_solver* s) {
    Crowd& c = crowd();
    std::lock_guard<std::mutex> lock(c.m);
    try {
        c.members.push_back(s);
    } catch (const std::bad_alloc&) {
        return fail(FVLBM_ERR_OOM, "fvlbm_init: out of host memory");
    }
    s->member = true;
    return FVLBM_OK;
}
static void crowd_leave(fvlbm_solver* s) {
    if (!s->member) return;
    Crowd& c = crowd();
    std::lock_guard<std::mutex> lock(c.m);
    c.members.erase(std::remove(c.members.begin(), c.members.end(), s), c.members.end());
}
// The solver's work is done.
static void crowd_idle(fvlbm_solver* s) {
    if (!s->member) return;
    std::lock_guard<std::mutex> lock(crowd().m);
    s->busy_until = 0;
}
static double crowd_now() {   // microseconds
    return std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now().time_since_epoch()).count();
}
// Whether the solver's next long call, of so many stages, runs in the resident loop.
static bool crowd_turns(fvlbm_solver* s, int64_t stages) {
    constexpr int QUEUES = 8;   // streams that CUDA runs side by side by default
    Crowd& c = crowd();
    std::lock_guard<std::mutex> lock(c.m);
    const uint64_t last = s->call;
    const bool joined = s->joined;
    s->call = ++c.calls;
    s->joined = false;
    OverlapGain gain;
    gain.add(s->cost);
    const double now = crowd_now();
    for (fvlbm_solver* o : c.members) {
        if (o == s || o->device != s->device || o->stream == s->stream) continue;
        const bool busy = o->busy_until > now;
        if (busy) o->joined = true;
        if (busy || (joined && o->call > last)) gain.add(o->cost);
    }
    const double in_turns = gain.in_turns(), overlapping = gain.overlapping(QUEUES), more = in_turns - overlapping;
    bool turns = more <= 0;
    if (!turns && !s->gk[0] && !s->gk[1] && s->lost < gain.n * GRAPH_SETUP_US) {
        s->lost += more * stages;
        turns = true;
    }
    s->busy_until = std::max(now, s->busy_until) + stages * (turns ? std::max(in_turns, s->cost.alone) : overlapping);
    return turns;
}

namespace fvlbm {
void OverlapGain::add(const StageCost& x) {
    n++;
    base = std::max(base, x.base);
    flow += x.flow;
    if (x.resident) {
        turns += x.turn;
    } else {   // runs stage kernels in any case
        left_base = std::max(left_base, x.base);
        left_flow += x.flow;
    }
}
}  // namespace fvlbm

static int init_impl(const fvlbm_mesh* mesh, const fvlbm_params* params, int32_t n_params, void* stream,
                     void* workspace, size_t workspace_bytes, fvlbm_solver* s) {
    const Mesh& M = mesh->m;
    int rc = check_params(M, params, n_params);
    if (rc) return rc;
    const fvlbm_params& p0 = params[0];
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0)
        return fail(FVLBM_ERR_UNSUPPORTED, "fvlbm_init: no CUDA device");
    if (p0.device < 0 || p0.device >= ndev) return fail(FVLBM_ERR_ARG, "fvlbm_init: device %d out of range", p0.device);
    DeviceGuard dg(p0.device);
    s->device = p0.device;
    s->stream = (cudaStream_t)stream;
    s->prec = p0.precision;
    s->scheme = p0.scheme;
    s->n_cell = M.n_owned;
    s->n_inst = M.n_inst;
    s->inst_begin = M.inst_begin;
    int pageable = 0;
    if (cudaDeviceGetAttribute(&pageable, cudaDevAttrPageableMemoryAccess, p0.device) != cudaSuccess) {
        cudaGetLastError();
        pageable = 0;
    }
    s->host_can_direct = pageable == 1;
    s->host_direct = s->host_can_direct;

    // per-instance constants and the time step of Eqs. (CFL), (timetau)
    s->inst.resize(M.n_inst);
    for (int32_t k = 0; k < M.n_inst; k++) {
        const fvlbm_params& p = params[n_params == 1 ? 0 : k];
        InstParam& I = s->inst[k];
        std::memset(&I, 0, sizeof I);
        const double umax = instance_umax(M, k, p);
        double dt = p.dt > 0 ? p.dt : suggest_dt(M, k, p.tau, p.cfl > 0 ? p.cfl : 0.5, umax, p.scheme);
        const double cap = p.scheme == FVLBM_AB2 ? p.tau : 2.0 * p.tau;
        if (dt > cap * (1 + 1e-12))
            return fail(FVLBM_ERR_UNSTABLE_DT, "instance %d: dt = %g exceeds the collision limit %g", k, dt, cap);
        const double cfl = dt * (std::sqrt(2.0) + umax) / M.inst_cfl_len[k];
        if (cfl > 1.0 + 1e-12)
            return fail(FVLBM_ERR_UNSTABLE_DT, "instance %d: dt = %g gives CFL %g > 1", k, dt, cfl);
        I.tau = p.tau;
        I.inv_tau = 1.0 / p.tau;
        I.dt = dt;
        I.inv_tau_f = (float)I.inv_tau;
        I.dt_f = (float)dt;
        I.rho0 = p.rho0;
        I.u0x = p.u0[0];
        I.u0y = p.u0[1];
        for (int a = 0; a < FVLBM_Q; a++) {
            float sc = 1.0f;
            if (p.precision == FVLBM_FP16_DEV) {
                // power-of-two scale of the stored non-equilibrium part: an
                // estimate of |g_a - g^eq_a| from the size of the equilibrium
                // deviation maps to ~2^5, 2^11 below FP16's largest finite value:
                // the non-equilibrium part grows like tau |e . grad f^eq|, and
                // near the lid corners of a Re 10 cavity it reached 17 times the
                // estimate (with the estimate at ~2^12 such values saturated).
                // FP16 precision is relative down to 2^-14 (6e-5); below, the
                // step stays 2^-24 / scale (~2e-10 of n here)
                const double w = a == 0 ? 4.0 / 9 : (a < 5 ? 1.0 / 9 : 1.0 / 36);
                const double e = a == 0 ? 0.0 : (a < 5 ? 1.0 : std::sqrt(2.0));
                const double U = std::max(umax, 1e-3);
                const double gmax = w * (0.1 + 2.2 * (3 * e * U + 4.5 * e * e * U * U + 1.5 * U * U));
                sc = std::ldexp(1.0f, (int)std::floor(std::log2(32.0 / gmax)));
            }
            I.scale[a] = sc;
            I.inv_scale[a] = 1.0f / sc;
        }
    }

    // layout, workspace
    Layout L;
    try {
        rc = make_layout(*mesh, s->prec, s->scheme, p0.kernel, L, device_sms(p0.device));
        // a workspace that holds everything but the loop's arrays is enough
        if (!rc && workspace && workspace_bytes < L.total && L.resident)
            rc = make_layout(*mesh, s->prec, s->scheme, p0.kernel, L, device_sms(p0.device), false, false);
    } catch (const std::bad_alloc&) {
        return fail(FVLBM_ERR_OOM, "fvlbm_init: out of host memory");
    }
    if (rc) return rc;
    if (workspace) {
        if (workspace_bytes < L.total)
            return fail(FVLBM_ERR_OOM, "fvlbm_init: workspace of %zu bytes, %zu needed", workspace_bytes, L.total);
        if ((uintptr_t)workspace % ALIGN) return fail(FVLBM_ERR_ARG, "fvlbm_init: workspace not 256-byte aligned");
        s->ws = workspace;
        s->own_ws = false;
    } else {
        cudaError_t e = cudaMalloc(&s->ws, L.total);
        if (e != cudaSuccess) {
            s->ws = nullptr;
            return fail(FVLBM_ERR_OOM, "fvlbm_init: cudaMalloc(%zu): %s", L.total, cudaGetErrorString(e));
        }
        s->own_ws = true;
    }
    s->ws_bytes = L.total;

    // host image of the read-only part (geometry, params, chunk table)
    std::vector<unsigned char> host;
    try {
        host.assign(L.off_fa, 0);
        if (s->prec == FVLBM_FP64) pack_geometry<double>(M, L, host);
        else pack_geometry<float>(M, L, host);
    } catch (const std::bad_alloc&) {
        return fail(FVLBM_ERR_OOM, "fvlbm_init: out of host memory");
    }
    std::memcpy(host.data() + L.off_inst, s->inst.data(), sizeof(InstParam) * M.n_inst);
    BcParam* bcp = (BcParam*)(host.data() + L.off_bc);
    for (size_t b = 0; b < M.bcs.size(); b++) {
        const fvlbm_bc& c = M.bcs[b];
        BcParam& q = bcp[b];
        q.kind = c.kind == FVLBM_BC_WALL ? SK_WALL : c.kind == FVLBM_BC_INLET ? SK_INLET
               : c.kind == FVLBM_BC_OUTLET ? SK_OUTLET : c.kind == FVLBM_BC_SYMMETRY ? SK_SYMMETRY : SK_NONE;
        q.external = c.external;
        q.uwx = c.u_w[0];
        q.uwy = c.u_w[1];
        q.rho_inf = c.rho_inf;
        q.uix = c.u_inf[0];
        q.uiy = c.u_inf[1];
        q.uwx_f = (float)q.uwx;
        q.uwy_f = (float)q.uwy;
        q.rho_f = (float)q.rho_inf;
        q.rdev_f = (float)(q.rho_inf - 1.0);
        q.uix_f = (float)q.uix;
        q.uiy_f = (float)q.uiy;
    }
    std::vector<int64_t> chunks, inst_chunk(1, 0);
    for (int32_t k = 0; k < M.n_inst; k++) {
        for (int64_t b = M.inst_begin[k]; b < M.inst_begin[k + 1]; b += CHUNK)
            chunks.insert(chunks.end(), {b, std::min(b + CHUNK, M.inst_begin[k + 1]), (int64_t)k});
        inst_chunk.push_back((int64_t)chunks.size() / 3);
    }
    const int64_t n_chunk = inst_chunk.back();
    chunks.insert(chunks.end(), inst_chunk.begin(), inst_chunk.end());

    unsigned char* base = (unsigned char*)s->ws;
    CK(cudaMemcpyAsync(base, host.data(), L.off_fa, cudaMemcpyHostToDevice, s->stream), "upload geometry");
    CK(cudaMemcpyAsync(base + L.off_chunk, chunks.data(), chunks.size() * sizeof(int64_t), cudaMemcpyHostToDevice,
                       s->stream), "upload chunk table");
    CK(cudaMemsetAsync(base + L.off_flag, 0, 16, s->stream), "clear flag");

    DevView& v = s->v;
    v.n_cell = M.n_owned;
    v.n_grad = M.n_grad;
    v.n_bface = M.n_bface;
    v.np = L.np;
    v.maxf = L.maxf;
    v.n_inst = M.n_inst;
    v.link = (const uint4*)(base + L.off_link);
    v.geo = base + L.off_geo;
    v.bctag = (const uint16_t*)(base + L.off_bctag);
    v.nbr = (const int4*)(base + L.off_nbr);
    v.area = (const double*)(base + L.off_area);
    v.grp = (const int32_t*)(base + L.off_grp);
    v.iperm = (const int32_t*)(base + L.off_iperm);
    v.inst = (const InstParam*)(base + L.off_inst);
    v.bc = (const BcParam*)(base + L.off_bc);
    v.fa = base + L.off_fa;
    v.fb = L.off_fb ? base + L.off_fb : nullptr;
    v.rprev = L.off_rprev ? base + L.off_rprev : nullptr;
    v.fv = base + L.off_fv;
    v.uold = (double*)(base + L.off_uold);
    v.part = (double*)(base + L.off_part);
    v.red = (double*)(base + L.off_red);
    v.conv = (double*)(base + L.off_conv);
    v.chunk = (const int64_t*)(base + L.off_chunk);
    v.n_chunk = n_chunk;
    v.inst_chunk = v.chunk + 3 * n_chunk;
    v.flag = (int32_t*)(base + L.off_flag);
    v.strategy = L.strategy;
    v.block = L.block;
    if (L.strategy == STRATEGY_TILE) {
        v.tile = L.tp.tile;
        v.tile_ghosts = L.tp.max_ghosts;
        v.n_tiles = L.tp.n_tiles;
        v.tiles = (const TileRec*)(base + L.off_tiles);
        v.halo = (const int32_t*)(base + L.off_halo);
        v.r1link = (const uint4*)(base + L.off_r1link);
        v.n_r1 = L.tp.n_r1;
    }
    v.sms = device_sms(p0.device);
    if (L.resident) {
        ResView& r = s->res;
        r.tile = L.res_plan().tile;
        r.n_tiles = (int32_t)L.res_plan().n_tiles;
        r.tiles = (const TileRec*)(base + L.off_rtiles);
        r.link = (const uint4*)(base + L.off_rlink);
        r.halo = (const int32_t*)(base + L.off_rhalo);
        r.r1link = (const uint4*)(base + L.off_rr1link);
        r.n_r1 = L.res_plan().n_r1;
        r.xchg = (uint4*)(base + L.off_xchg);
        CK(cudaMemsetAsync(r.xchg, 0, 2 * 16 * (size_t)resident_units(state_bytes(s->prec)) * L.np, s->stream), "clear tags");
        const int max_ctas = resident_max_ctas(v, r, s->prec, s->scheme);
        s->resident = max_ctas >= r.n_tiles;
        if (s->resident) s->cost = stage_cost(v, s->prec, &r, max_ctas);
    }
    if (!s->resident) s->cost = stage_cost(v, s->prec, nullptr, 0);
    if (s->resident) {
        rc = crowd_join(s);
        if (rc) return rc;
    }
    s->pingpong = L.pingpong;
    s->buf[0] = v.fa;
    s->buf[1] = v.fb;
    s->fc = L.off_fc ? base + L.off_fc : nullptr;
    s->cur = 0;

    // Step 0 and the first residual snapshot
    rc = launch_init_eq(v, s->prec, s->stream);
    if (rc) return rc;
    rc = launch_snapshot(v, s->prec, s->stream);
    if (rc) return rc;
    CK(cudaStreamSynchronize(s->stream), "fvlbm_init");
    return FVLBM_OK;
}

extern "C" void fvlbm_solver_destroy(fvlbm_solver* s) {
    if (!s) return;
    crowd_leave(s);
    for (int b = 0; b < 2; b++) {
        if (s->g1[b]) cudaGraphExecDestroy(s->g1[b]);
        if (s->gk[b]) cudaGraphExecDestroy(s->gk[b]);
    }
    if (s->own_ws && s->ws) {
        DeviceGuard dg(s->device);
        cudaStreamSynchronize(s->stream);
        cudaFree(s->ws);
    }
    delete s;
}

extern "C" int fvlbm_init(const fvlbm_mesh* mesh, const fvlbm_params* params, int32_t n_params, void* stream,
                          void* workspace, size_t workspace_bytes, fvlbm_solver** out) {
    clear_error();
    if (!mesh || !out) return fail(FVLBM_ERR_ARG, "fvlbm_init: null argument");
    *out = nullptr;
    fvlbm_solver* s = new (std::nothrow) fvlbm_solver;
    if (!s) return fail(FVLBM_ERR_OOM, "fvlbm_init: out of host memory");
    int rc = init_impl(mesh, params, n_params, stream, workspace, workspace_bytes, s);
    if (rc != FVLBM_OK) {
        fvlbm_solver_destroy(s);
        return rc;
    }
    *out = s;
    return FVLBM_OK;
}

// Stages per time step of each scheme.
static int n_stages(int scheme) { return scheme == FVLBM_RK2 ? 2 : scheme == FVLBM_RK4 ? 4 : 1; }

// Make buf[c] the current state (v.fa) and the other buffer v.fb.
static void set_current(fvlbm_solver* s, int c) {
    s->cur = c;
    s->v.fa = s->buf[c];
    s->v.fb = s->buf[c ^ 1];
}

// Enqueue stage k of one time step (0 <= k < n_stages).  ev: null, or 3
// events (see launch_stage).  *out (if not null): the buffer the stage writes.
// The last stage of a single-stage scheme also ends the step (AB2 history,
// alternating state).
static int enqueue_stage(fvlbm_solver* s, int k, void* const* ev, void** out) {
    const DevView& v = s->v;
    void* dst = nullptr;
    int rc = FVLBM_OK;
    switch (s->scheme) {
        case FVLBM_EULER:
        case FVLBM_AB2: {
            const int mode = s->scheme == FVLBM_EULER ? MODE_RK : (s->ab2_started ? MODE_AB2 : MODE_AB2_FIRST);
            // in place on the two-kernel stage (each cell reads only its own state
            // after the face values are written); fa -> fb and swap on the fused stage
            dst = s->pingpong ? v.fb : v.fa;
            rc = launch_stage(v, s->prec, s->stream, v.fa, v.fa, dst, 1.0, mode, ev);
            if (rc) return rc;
            if (s->scheme == FVLBM_AB2) s->ab2_started = true;
            if (s->pingpong) set_current(s, s->cur ^ 1);
            break;
        }
        case FVLBM_RK2:
            dst = k == 0 ? v.fb : v.fa;
            rc = launch_stage(v, s->prec, s->stream, k == 0 ? v.fa : v.fb, v.fa, dst, k == 0 ? 0.5 : 1.0, MODE_RK, ev);
            break;
        case FVLBM_RK4: {
            static const double beta[4] = {0.25, 1.0 / 3.0, 0.5, 1.0};
            // fa -> fb -> fb -> fb -> fa, or with a third buffer fa -> fb -> fc -> fb -> fa
            void* const in[4] = {v.fa, v.fb, s->fc ? s->fc : v.fb, v.fb};
            void* const o[4] = {v.fb, s->fc ? s->fc : v.fb, v.fb, v.fa};
            dst = o[k];
            rc = launch_stage(v, s->prec, s->stream, in[k], v.fa, dst, beta[k], MODE_RK, ev);
            break;
        }
        default:
            return fail(FVLBM_ERR_ARG, "bad scheme");
    }
    if (out) *out = dst;
    return rc;
}

// Enqueue one time step.  ev: null, or 3 events per stage (see launch_stage).
static int enqueue_step(fvlbm_solver* s, void* const* ev = nullptr) {
    const int ns = n_stages(s->scheme);
    for (int k = 0; k < ns; k++) {
        int rc = enqueue_stage(s, k, ev ? ev + 3 * k : ev, nullptr);
        if (rc) return rc;
    }
    return FVLBM_OK;
}

extern "C" int fvlbm_profile(fvlbm_solver* s, int64_t n, double* avg_ms, int32_t max_kinds, int32_t* n_kinds,
                             int64_t* launches) {
    clear_error();
    if (!s || n <= 0 || !avg_ms || max_kinds < STAGE_KERNELS || !n_kinds || !launches)
        return fail(FVLBM_ERR_ARG, "fvlbm_profile: bad arguments");
    DeviceGuard dg(s->device);
    const int ns = n_stages(s->scheme);
    std::vector<cudaEvent_t> ev((size_t)3 * ns * n, nullptr);
    int rc = FVLBM_OK;
    for (auto& e : ev) {
        cudaError_t ce = cudaEventCreate(&e);
        if (ce != cudaSuccess) {
            e = nullptr;
            rc = cuda_fail(ce, "fvlbm_profile: event");
            break;
        }
    }
    for (int64_t k = 0; k < n && rc == FVLBM_OK; k++) rc = enqueue_step(s, (void* const*)&ev[(size_t)3 * ns * k]);
    if (rc == FVLBM_OK) {
        cudaError_t ce = cudaStreamSynchronize(s->stream);
        if (ce != cudaSuccess) rc = cuda_fail(ce, "fvlbm_profile: synchronise");
    }
    if (rc == FVLBM_OK) {
        double t[STAGE_KERNELS] = {0, 0};
        for (size_t q = 0; q < ev.size(); q += 3) {
            float a = 0, b = 0;
            cudaEventElapsedTime(&a, ev[q], ev[q + 1]);
            cudaEventElapsedTime(&b, ev[q + 1], ev[q + 2]);
            t[0] += a;
            t[1] += b;
        }
        const double launches_per_kind = (double)ns * n;
        const int kinds = stage_kernels(s->v);
        for (int q = 0; q < kinds; q++) avg_ms[q] = t[q] / launches_per_kind;
        *n_kinds = kinds;
        *launches = (int64_t)kinds * ns * n;
    }
    for (auto& e : ev)
        if (e) cudaEventDestroy(e);
    return rc;
}

extern "C" int fvlbm_launches_per_step(const fvlbm_solver* s, int64_t* launches) {
    clear_error();
    if (!s || !launches) return fail(FVLBM_ERR_ARG, "fvlbm_launches_per_step: null argument");
    *launches = (int64_t)stage_kernels(s->v) * n_stages(s->scheme);
    return FVLBM_OK;
}

// Capture `nsteps` steps of the solver's stream into an executable graph.
// Capture only records launches: the host-side state (current buffer, AB2
// start) is put back afterwards.
static bool build_graph(fvlbm_solver* s, int64_t nsteps, cudaGraphExec_t* out) {
    const int cur0 = s->cur;
    const bool ab2 = s->ab2_started;
    if (cudaStreamBeginCapture(s->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    int rc = FVLBM_OK;
    for (int64_t k = 0; k < nsteps && rc == FVLBM_OK; k++) rc = enqueue_step(s);
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(s->stream, &g);
    set_current(s, cur0);
    s->ab2_started = ab2;
    bool ok = rc == FVLBM_OK && e == cudaSuccess && g;
    if (ok) ok = cudaGraphInstantiate(out, g, 0) == cudaSuccess;
    if (g) cudaGraphDestroy(g);
    if (!ok) {
        *out = nullptr;
        cudaGetLastError();
        clear_error();
    }
    return ok;
}

// Steps are replayed from CUDA graphs (chunks of GRAPH_CHUNK, then single
// steps) once the solver has run directly at least once (so that kernel
// attributes are set outside capture) and AB2 has its history; the legacy
// default stream cannot be captured and always launches directly.  With a
// ping-pong state there is one pair of graphs per starting buffer (a chunk
// has an even number of steps and ends where it started).
extern "C" int fvlbm_step(fvlbm_solver* s, int64_t n) {
    clear_error();
    if (!s || n < 0) return fail(FVLBM_ERR_ARG, "fvlbm_step: bad arguments");
    DeviceGuard dg(s->device);
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(s->stream, &cs);
    bool graphs = s->graphs_ok && s->stream != nullptr && cs == cudaStreamCaptureStatusNone &&
                  s->direct_steps > 0 && (s->scheme != FVLBM_AB2 || s->ab2_started);
    // small solvers: chunks of whole steps, at least two stages each, in the
    // resident loop (a caller's capture records the stages one by one).  Calls shorter
    // than a graph's steps are bound by the host's launches, of which the loop makes fewer
    const bool in_crowd = s->resident && s->path == STEP_AUTO && s->stream && cs == cudaStreamCaptureStatusNone && n >= GRAPH_CHUNK;
    const bool turns = s->path == STEP_AUTO ? !in_crowd || crowd_turns(s, n * n_stages(s->scheme)) : s->path == STEP_RESIDENT;
    if (s->resident && turns && cs == cudaStreamCaptureStatusNone) {
        const int ns = n_stages(s->scheme);
        while (n * ns >= 2) {
            int64_t m = std::min(n, RESIDENT_CHUNK / ns);
            if ((n - m) * ns == 1) m--;
            int rc = launch_resident(s->v, s->res, s->prec, s->stream, s->scheme, m * ns, s->epoch, s->ab2_started);
            if (rc == FVLBM_ERR_UNSUPPORTED) {   // from here on the stage kernels, which need no such room
                clear_error();
                s->resident = false;
                break;
            }
            if (rc) return rc;
            s->res_launches++;
            s->epoch += (uint32_t)(m * ns);
            s->ab2_started = s->scheme == FVLBM_AB2;
            n -= m;
        }
    }
    auto ready = [&](int b) {
        if (s->g1[b]) return true;
        if (!build_graph(s, 1, &s->g1[b]) || !build_graph(s, GRAPH_CHUNK, &s->gk[b])) {
            s->graphs_ok = false;
            return false;
        }
        return true;
    };
    while (n > 0) {
        if (graphs && !ready(s->cur)) graphs = false;
        int rc = FVLBM_OK;
        if (graphs && n >= GRAPH_CHUNK) {
            cudaError_t e = cudaGraphLaunch(s->gk[s->cur], s->stream);
            if (e != cudaSuccess) return cuda_fail(e, "fvlbm_step: graph launch");
            n -= GRAPH_CHUNK;
            continue;
        }
        if (graphs) {
            cudaError_t e = cudaGraphLaunch(s->g1[s->cur], s->stream);
            rc = e == cudaSuccess ? FVLBM_OK : cuda_fail(e, "fvlbm_step: graph launch");
            if (rc == FVLBM_OK && s->pingpong) set_current(s, s->cur ^ 1);
        } else {
            rc = enqueue_step(s);
            s->direct_steps++;
        }
        if (rc) return rc;
        n--;
    }
    return FVLBM_OK;
}

static int sync_and_check(fvlbm_solver* s) {
    int32_t flag[2] = {0, 0};
    CK(cudaMemcpyAsync(flag, s->v.flag, sizeof flag, cudaMemcpyDeviceToHost, s->stream), "read flag");
    CK(cudaStreamSynchronize(s->stream), "synchronise");
    crowd_idle(s);
    if (flag[1]) return fail(FVLBM_ERR_TIMEOUT, "the resident stage loop: a tile waited too long for its neighbours");
    if (flag[0]) return fail(FVLBM_ERR_DIVERGED, "a non-finite value appeared in the state");
    return FVLBM_OK;
}

namespace fvlbm {
int solver_ref(fvlbm_solver* s, SolverRef* out) {
    if (!s || !out) return fail(FVLBM_ERR_ARG, "null solver");
    out->view = &s->v;
    out->prec = s->prec;
    out->device = s->device;
    out->stream = s->stream;
    out->n_inst = s->n_inst;
    return FVLBM_OK;
}
int solver_sync_check(fvlbm_solver* s) { return sync_and_check(s); }
}  // namespace fvlbm

extern "C" int fvlbm_sync(fvlbm_solver* s) {
    clear_error();
    if (!s) return fail(FVLBM_ERR_ARG, "fvlbm_sync: null solver");
    DeviceGuard dg(s->device);
    return sync_and_check(s);
}

extern "C" int fvlbm_macros(fvlbm_solver* s, double* rho, double* u) {
    clear_error();
    if (!s) return fail(FVLBM_ERR_ARG, "fvlbm_macros: null solver");
    DeviceGuard dg(s->device);
    // caller order in the device staging buffer, then one copy per output
    // (device -> host always staged; see fvlbm_host_transfer)
    double* d_rho = s->v.conv;
    double* d_u = s->v.conv + s->n_cell;
    int rc = launch_macros_ordered(s->v, s->prec, s->stream, rho ? d_rho : nullptr, u ? d_u : nullptr);
    if (rc) return rc;
    // cudaMemcpyDefault: the caller's buffer may be host (pageable or pinned) or device memory
    if (rho) CK(cudaMemcpyAsync(rho, d_rho, 8 * (size_t)s->n_cell, cudaMemcpyDefault, s->stream), "read rho");
    if (u) CK(cudaMemcpyAsync(u, d_u, 16 * (size_t)s->n_cell, cudaMemcpyDefault, s->stream), "read u");
    return sync_and_check(s);
}

static int reduce(fvlbm_solver* s, int what, std::vector<double>& out) {
    int rc = launch_reduce(s->v, s->prec, s->stream, what);
    if (rc) return rc;
    out.assign(2 * (size_t)s->n_inst, 0.0);
    CK(cudaMemcpyAsync(out.data(), s->v.red, out.size() * 8, cudaMemcpyDeviceToHost, s->stream), "read sums");
    return sync_and_check(s);
}

namespace fvlbm {
int solver_n_stages(const fvlbm_solver* s) { return n_stages(s->scheme); }
int solver_stage(fvlbm_solver* s, int k, void** out) {
    if (!s || k < 0 || k >= n_stages(s->scheme)) return fail(FVLBM_ERR_ARG, "solver_stage: bad arguments");
    DeviceGuard dg(s->device);
    s->staged = true;
    return enqueue_stage(s, k, nullptr, out);
}
bool solver_replayable(const fvlbm_solver* s) {
    return s->staged && (s->scheme != FVLBM_AB2 || s->ab2_started);
}
int solver_buffer(const fvlbm_solver* s) { return s->cur; }
void solver_set_buffer(fvlbm_solver* s, int b) { set_current(s, b); }
StageCost solver_cost(const fvlbm_solver* s) { return s->cost; }
double solver_overlap_setup(const fvlbm_solver* s) { return s->gk[0] || s->gk[1] ? 0.0 : request_setup_us(s->prec); }
void solver_path(fvlbm_solver* s, StepPath path) { s->path = path; }
int solver_sums(fvlbm_solver* s, int what, std::vector<double>& out) {
    DeviceGuard dg(s->device);
    return reduce(s, what, out);
}
}  // namespace fvlbm

extern "C" int fvlbm_residual(fvlbm_solver* s, double* e) {
    clear_error();
    if (!s || !e) return fail(FVLBM_ERR_ARG, "fvlbm_residual: null argument");
    DeviceGuard dg(s->device);
    std::vector<double> r;
    int rc = reduce(s, RED_RESIDUAL, r);
    if (rc) return rc;
    for (int32_t k = 0; k < s->n_inst; k++) {
        const double num = r[2 * k], den = r[2 * k + 1];
        e[k] = den == 0 ? (num == 0 ? 0.0 : INFINITY) : std::sqrt(num) / std::sqrt(den);
    }
    return FVLBM_OK;
}

extern "C" int fvlbm_mass(fvlbm_solver* s, double* mass) {
    clear_error();
    if (!s || !mass) return fail(FVLBM_ERR_ARG, "fvlbm_mass: null argument");
    DeviceGuard dg(s->device);
    std::vector<double> r;
    int rc = reduce(s, RED_MASS, r);
    if (rc) return rc;
    for (int32_t k = 0; k < s->n_inst; k++) mass[k] = r[2 * k];
    return FVLBM_OK;
}

extern "C" int fvlbm_get_f(fvlbm_solver* s, double* f) {
    clear_error();
    if (!s || !f) return fail(FVLBM_ERR_ARG, "fvlbm_get_f: null argument");
    DeviceGuard dg(s->device);
    // caller order in the device staging buffer, then one copy (device -> host
    // always staged; see fvlbm_host_transfer)
    int rc = launch_get_f_ordered(s->v, s->prec, s->stream, s->v.conv);
    if (rc) return rc;
    CK(cudaMemcpyAsync(f, s->v.conv, 8 * (size_t)s->n_cell * FVLBM_Q, cudaMemcpyDefault, s->stream), "read f");
    return sync_and_check(s);
}

extern "C" int fvlbm_set_f(fvlbm_solver* s, const double* f) {
    clear_error();
    if (!s || !f) return fail(FVLBM_ERR_ARG, "fvlbm_set_f: null argument");
    DeviceGuard dg(s->device);
    CK(cudaStreamSynchronize(s->stream), "synchronise");
    int rc;
    if (s->host_direct) {
        rc = launch_set_f_ordered(s->v, s->prec, s->stream, f);
    } else {
        // staged: one copy of the caller's buffer into the device staging buffer
        CK(cudaMemcpyAsync(s->v.conv, f, 8 * (size_t)s->n_cell * FVLBM_Q, cudaMemcpyDefault, s->stream), "write f");
        rc = launch_set_f_ordered(s->v, s->prec, s->stream, s->v.conv);
    }
    if (rc) return rc;
    s->ab2_started = false;
    if (s->scheme == FVLBM_AB2) s->direct_steps = 0;   // the next step is an Euler start, launched directly
    CK(cudaStreamSynchronize(s->stream), "synchronise");
    return FVLBM_OK;
}

extern "C" int fvlbm_stage_kernel(const fvlbm_solver* s, int32_t* kernel) {
    clear_error();
    if (!s || !kernel) return fail(FVLBM_ERR_ARG, "fvlbm_stage_kernel: null argument");
    *kernel = s->v.strategy == STRATEGY_TILE ? s->v.tile : 1;
    return FVLBM_OK;
}

extern "C" int fvlbm_resident_info(const fvlbm_solver* s, int32_t* tile, int32_t* tiles, int64_t* launches) {
    clear_error();
    if (!s) return fail(FVLBM_ERR_ARG, "fvlbm_resident_info: null solver");
    if (tile) *tile = s->resident ? s->res.tile : 0;
    if (tiles) *tiles = s->resident ? s->res.n_tiles : 0;
    if (launches) *launches = s->res_launches;
    return FVLBM_OK;
}

extern "C" int fvlbm_resident_polls(fvlbm_solver* s, int32_t polls) {
    clear_error();
    if (!s || polls < 0) return fail(FVLBM_ERR_ARG, "fvlbm_resident_polls: bad arguments");
    s->res.polls = polls;
    return FVLBM_OK;
}

extern "C" int fvlbm_host_transfer(fvlbm_solver* s, int32_t mode, int32_t* direct) {
    clear_error();
    if (!s || (mode != FVLBM_HOST_AUTO && mode != FVLBM_HOST_STAGED))
        return fail(FVLBM_ERR_ARG, "fvlbm_host_transfer: bad arguments");
    s->host_direct = mode == FVLBM_HOST_AUTO && s->host_can_direct;
    if (direct) *direct = s->host_direct ? 1 : 0;
    return FVLBM_OK;
}

extern "C" int fvlbm_get_dt(const fvlbm_solver* s, int32_t instance, double* dt) {
    clear_error();
    if (!s || !dt || instance < 0 || instance >= s->n_inst) return fail(FVLBM_ERR_ARG, "fvlbm_get_dt: bad arguments");
    *dt = s->inst[instance].dt;
    return FVLBM_OK;
}

extern "C" int fvlbm_autotune(const fvlbm_mesh* mesh, const fvlbm_params* params, int32_t n_params, void* stream,
                              int32_t steps, int32_t* best_kernel, double* ms_per_step) {
    clear_error();
    if (!mesh || !params || n_params <= 0 || steps <= 0 || !best_kernel)
        return fail(FVLBM_ERR_ARG, "fvlbm_autotune: bad arguments");
    static const int32_t cand[5] = {1, 128, 256, 512, 1024};
    constexpr int REPEATS = 5;
    std::vector<fvlbm_params> p(params, params + n_params);
    double med[5];
    // the automatic choice (params.kernel = 0) for this mesh
    int32_t automatic = 0;
    {
        Layout L;
        if (make_layout(*mesh, params[0].precision, params[0].scheme, 0, L, device_sms(params[0].device)) == FVLBM_OK)
            automatic = L.strategy == STRATEGY_TILE ? L.tp.tile : 1;
        clear_error();
    }
    for (int c = 0; c < 5; c++) {
        med[c] = INFINITY;
        for (auto& q : p) q.kernel = cand[c];
        fvlbm_solver* sv = nullptr;
        int rc = fvlbm_init(mesh, p.data(), n_params, stream, nullptr, 0, &sv);
        if (rc == FVLBM_ERR_UNSUPPORTED || rc == FVLBM_ERR_OOM) continue;   // variant does not fit
        if (rc) return rc;
        DeviceGuard dg(sv->device);
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        rc = fvlbm_step(sv, 3);   // warm-up: direct launches, then the graphs are built
        if (!rc) rc = fvlbm_sync(sv);
        if (!rc && (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess))
            rc = fail(FVLBM_ERR_CUDA, "fvlbm_autotune: events");
        double t[REPEATS];
        for (int r = 0; r < REPEATS && !rc; r++) {
            float ms = 0;
            cudaEventRecord(e0, sv->stream);
            rc = fvlbm_step(sv, steps);
            cudaEventRecord(e1, sv->stream);
            if (!rc) rc = fvlbm_sync(sv);
            if (!rc) cudaEventElapsedTime(&ms, e0, e1);
            t[r] = ms / steps;
        }
        if (e0) cudaEventDestroy(e0);
        if (e1) cudaEventDestroy(e1);
        fvlbm_solver_destroy(sv);
        if (rc) return rc;
        std::sort(t, t + REPEATS);
        med[c] = t[REPEATS / 2];
    }
    int best = -1;
    for (int c = 0; c < 5; c++)
        if (std::isfinite(med[c]) && (best < 0 || med[c] < med[best])) best = c;
    if (best < 0) return fail(FVLBM_ERR_UNSUPPORTED, "fvlbm_autotune: no stage kernel variant fits");
    // timing noise must not flip the choice between variants that are as fast:
    // among those within 3% (or 2 microseconds per step, the launch jitter that
    // small meshes see) of the fastest median, the automatic choice wins, else
    // the first in a fixed order
    static const int32_t pref[5] = {512, 256, 128, 1024, 1};
    const double lim = std::max(1.03 * med[best], med[best] + 0.002);
    int pick = -1;
    for (int c = 0; c < 5; c++)
        if (cand[c] == automatic && med[c] <= lim) pick = c;
    for (int q = 0; q < 5 && pick < 0; q++)
        for (int c = 0; c < 5; c++)
            if (cand[c] == pref[q] && med[c] <= lim) pick = c;
    best = pick;
    if (ms_per_step)
        for (int c = 0; c < 5; c++) ms_per_step[c] = med[c];
    *best_kernel = cand[best];
    return FVLBM_OK;
}
