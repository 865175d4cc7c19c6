// Internal declarations shared by the host side (mesh, solver) and the CUDA
// kernels of the library.  Not part of the public ABI.
#pragma once

#include <cstdint>
#include <cstddef>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include <cuda_runtime_api.h>
#include <vector_types.h>

#include "fvlbm.h"

namespace fvlbm {

// Makes device d current for the guard's scope and restores the caller's
// device afterwards (also when the caller's device could not be read: then the
// device is left as the scope set it, as no previous one is known).
struct DeviceGuard {
    int prev = -1;
    bool ok = true;   // device d is current
    explicit DeviceGuard(int d) {
        if (cudaGetDevice(&prev) != cudaSuccess) {
            cudaGetLastError();
            prev = -1;
        }
        if (prev != d && cudaSetDevice(d) != cudaSuccess) {
            cudaGetLastError();
            ok = false;
        }
    }
    ~DeviceGuard() {
        int cur;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
    DeviceGuard(const DeviceGuard&) = delete;
    DeviceGuard& operator=(const DeviceGuard&) = delete;
};

// ---------------------------------------------------------------- errors
// Records a message for fvlbm_last_error() and returns `code`.
int fail(int code, const char* fmt, ...);
void clear_error();

// ---------------------------------------------------------------- mesh (host, FP64)
// Face-slot kinds as the kernels see them.
enum SlotKind : uint32_t {
    SK_NONE = 0,      // unused slot (cell has fewer faces)
    SK_INTERIOR = 1,  // interior or periodic face: neighbour cell across it
    SK_WALL = 2,
    SK_INLET = 3,
    SK_OUTLET = 4,
    SK_SYMMETRY = 5,
};

struct Slot {
    int32_t kind = SK_NONE;  // SlotKind
    int32_t nb = -1;         // neighbour cell (caller numbering of the instance-local mesh)
    int32_t nb_slot = -1;    // the same face's slot inside the neighbour
    int32_t bc = -1;         // boundary tag (boundary slots)
    int32_t periodic = 0;    // 1 if the face is a periodic pair
    double nx = 0, ny = 0;   // outward normal times length: (dy, -dx) of the CCW edge
    double px = 0, py = 0;   // face midpoint
    double sx = 0, sy = 0;   // periodic: neighbour image = neighbour centroid + (sx, sy)
    double cgx = 0, cgy = 0; // least-squares coefficient of this slot's stencil point
    double vx = 0, vy = 0;   // start vertex of the edge (the edge runs to the next slot's)
    double sdx = 0, sdy = 0; // stencil point minus cell centroid
    uint32_t outmask = 0;    // bit a-1 set when e_a . n > 0 (a = 1..8): upwind side is this cell
};

constexpr int MAXP = FVLBM_MAX_POLY;

struct Mesh {
    int64_t n_cell = 0;
    // A part of a partitioned mesh also holds ghost cells: cells [0, n_owned)
    // (the same in both numberings) are the part's own and are updated; cells
    // [n_owned, n_grad) are the first ghost ring (their gradient is recomputed
    // from local data), [n_grad, n_cell) the second (state only).  A whole
    // mesh has n_owned = n_grad = n_cell.
    int64_t n_owned = 0, n_grad = 0;
    int32_t max_faces = 0;
    int32_t n_inst = 1;
    std::vector<int64_t> inst_begin;     // [n_inst + 1] cell ranges (same in both numberings)
    std::vector<int32_t> inst_bc_begin;  // [n_inst + 1] ranges of bcs
    std::vector<fvlbm_bc> bcs;           // all boundary tags (global numbering)
    std::vector<double> inst_cfl_len;    // [n_inst] min A/(Lx+Ly)
    std::vector<int32_t> nf;             // [n_cell] faces per cell
    std::vector<double> area, cx, cy;    // [n_cell]
    std::vector<Slot> slots;             // [n_cell * MAXP]; nb is a global caller index
    std::vector<int64_t> perm;           // internal -> caller
    std::vector<int64_t> iperm;          // caller -> internal
    int64_t n_face = 0, n_bface = 0, n_periodic = 0;
    double total_area = 0;
};

// ---------------------------------------------------------------- device view
// Per-instance constants read by the kernels.
struct InstParam {
    double tau, inv_tau, dt;
    float inv_tau_f, dt_f;
    float scale[FVLBM_Q];      // 16-bit split storage: stored = (g_a - g^eq_a) * scale
    float inv_scale[FVLBM_Q];
    double rho0, u0x, u0y;
};

// Per-boundary-tag constants read by the kernels.
struct BcParam {
    int32_t kind;      // SlotKind of the tag
    int32_t external;
    double uwx, uwy, rho_inf, uix, uiy;
    // the same rounded to FP32 on the host (rdev_f = rho_inf - 1 in FP64,
    // then rounded), so that FP32 kernels do no FP64 arithmetic
    float uwx_f, uwy_f, rho_f, rdev_f, uix_f, uiy_f;
};

// Per-cell arrays on the device are blocked: 32 consecutive cells per block,
// each unit of the block contiguous (see blk_index in fvlbm_device.cuh).
constexpr int BLK_SHIFT = 5;
constexpr int BLK = 1 << BLK_SHIFT;

// Link word of one face slot of one cell:
//   bits  0..10  fused stage: tile-local index of the neighbour (the cell
//                itself for boundary and unused slots, so that the gradient
//                loop needs no test: the difference is zero)
//   bits 11..14  bit p set: direction A of pair p leaves the cell through this
//                face and B enters it (fvlbm_device.cuh), else the reverse.  The
//                two sides of a face hold complementary bits, which makes each
//                (face, direction) one side's to reconstruct
//   bits 15..17  LinkKind
//   bits 18..31  fused stage, tile cell: row of the tile's face table that
//                holds what enters through this face (the neighbour's outgoing
//                values, or the ghost values of a boundary face); two-kernel
//                stage: the same face's slot in the neighbour
enum LinkKind : uint32_t {
    LK_FLOW = 0,       // interior face
    LK_OTHER = 1,      // fused stage, 1-ring cell: a face the tile's cells do not have
    LK_WALL = 2,
    LK_INLET = 3,
    LK_OUTLET = 4,     // external-flow outlet
    LK_PRESSURE = 5,   // internal-flow (pressure) outlet
    LK_SYMMETRY = 6,
    LK_NONE = 7,       // unused slot (the cell has fewer faces)
};
constexpr uint32_t LINK_NB_MASK = 0x7FFu;
constexpr int LINK_PAIR_SHIFT = 11, LINK_KIND_SHIFT = 15, LINK_ROW_SHIFT = 18;
constexpr uint32_t LINK_ROW_MAX = 0x3FFFu;

// Fused stage: shared-memory capacity of a tile of TILE threads (compile-time
// strides, so that every shared-memory access is a fixed offset from one
// index): LS local cells (tile, 1-ring, 2-ring) and the face table, whose row
// k * TILE + x holds the four values that leave local cell x through slot k,
// and whose last GHOSTS rows hold the values that enter through the tile's
// boundary faces; reals of RSIZE bytes.  A row is one 16-byte unit in FP32, so that
// no offset depends on how many there are: tiles there have up to MAX_GHOSTS boundary
// faces, and a launch whose plan has tiles of more than GHOSTS asks for the memory
// (instances of a few cells, channels one cell wide: 30,000 meshes of two triangles 9.0 us
// per stage, 11.9 with tiles cut at GHOSTS).  The planner ends a tile early when it would
// not fit.
template <int TILE, int MAXF, int RSIZE> struct TileDims {
    static constexpr int LS = (3 * TILE) / 2 + 64;
    static constexpr int GHOSTS = TILE / 2;
    static constexpr int MAX_GHOSTS = RSIZE == 4 ? 2 * TILE : GHOSTS;
    static constexpr int ROWS = MAXF * TILE + GHOSTS;
    static constexpr size_t BYTES = (size_t)RSIZE * ((size_t)(FVLBM_Q - 1) * LS + (size_t)4 * ROWS);
    static constexpr size_t MAX_BYTES = BYTES + (size_t)4 * RSIZE * (MAX_GHOSTS - GHOSTS);
    static_assert(LS <= (int)LINK_NB_MASK + 1 && MAXF * TILE + MAX_GHOSTS <= (int)LINK_ROW_MAX, "link word fields");
};

// One tile of the fused stage.
struct TileRec {
    int32_t c0, nt;     // cells [c0, c0 + nt)
    int32_t h0, nh;     // halo entries [h0, h0 + nh): 1-ring, then 2-ring
    int32_t q0, n1;     // 1-ring entries [q0, q0 + n1) of the link array r1link
    int32_t inst;       // instance of every local cell, or -1 when they differ
    int32_t pad;
};

// Device pointers of one solver (all inside one workspace).
struct DevView {
    int64_t n_cell;     // cells updated (internal numbering 0..n_cell-1): the owned cells
    int64_t n_grad;     // cells whose gradient the two-kernel stage computes (owned + first ghost ring)
    int64_t n_bface;    // boundary faces of the cells
    int64_t np;         // padded cell count (multiple of the largest tile)
    int32_t maxf;       // slots per cell in the packed arrays (4 or 8)
    int32_t n_inst;
    // geometry, blocked per cell
    const uint4* link;     // [maxf / 4] units of four link words
    const void* geo;       // least-squares coefficients, face midpoint - centroid, face vector / area
                           // of each slot (GeoRef)
    const uint16_t* bctag; // [np][maxf] boundary tag of each slot (read for boundary slots only)
    // two-kernel stage: neighbour cell of interior slots, ghost record of boundary slots, the cell
    // itself for unused ones; blocked like link
    const int4* nbr;
    const double* area;    // [np]
    const int32_t* grp;    // [np] instance of each cell
    const int32_t* iperm;  // [n_cell] internal index of each cell in the caller's order
    const InstParam* inst; // [n_inst]
    const BcParam* bc;     // [n_bc]
    // state
    void* fa;   // blocked (PlainIO, SplitIO): the state
    void* fb;   // same: stage state (multistage schemes) or the other buffer of a ping-pong pair
    void* rprev;// T [9][np]  AB2 previous RHS
    void* fv;   // two-kernel stage: Quad<T> of outgoing values per (cell, slot), blocked [maxf], then the
                // ghost records (values that enter through boundary faces)
    double* uold;   // [2][np] the residual's snapshot of u
    double* part;   // [n_chunk][RED_PARTS][2] block partial sums
    double* red;    // [n_inst][2]  per-instance sums
    double* conv;   // [9][np] doubles: device staging of get_f / set_f / macros in caller order
    const int64_t* chunk;   // [n_chunk][3] (begin, end, instance)
    const int64_t* inst_chunk;   // [n_inst + 1] chunks of each instance
    int64_t n_chunk;
    int32_t* flag;  // [0] non-finite flag, [1] a wait of the resident kernel ran out
    // fused stage (one CTA per tile of at most `tile` consecutive cells)
    int32_t strategy;        // STRATEGY_TWO_KERNEL or STRATEGY_TILE
    int32_t block;           // threads per block of the two-kernel stage
    int32_t tile;            // most cells per tile (threads per CTA)
    int32_t tile_ghosts;     // most boundary faces of a tile
    int32_t sms;             // streaming multiprocessors of the device
    int64_t n_tiles;
    const TileRec* tiles;      // [n_tiles]
    const int32_t* halo;       // 1-ring then 2-ring cells of each tile (global ids)
    const uint4* r1link;       // [maxf / 4][n_r1] link words of the 1-ring entries
    int64_t n_r1;
};

// Most polls of a wait of the resident loop, of about half a microsecond: seconds,
// against microseconds of waiting.
constexpr int32_t RES_POLLS = 1 << 22;

// The resident plan of a small solver (fvlbm_resident.cuh): every tile has a
// CTA of its own on the GPU for as many time steps as one launch advances.
struct ResView {
    int32_t tile = 0;          // most tile and 1-ring cells of a tile (0: no resident plan)
    int32_t n_tiles = 0;
    const TileRec* tiles = nullptr;
    const uint4* link = nullptr;       // as DevView, in this plan's tiles
    const int32_t* halo = nullptr;
    const uint4* r1link = nullptr;
    int64_t n_r1 = 0;
    uint4* xchg = nullptr;             // [2][units][np] (FP64 [2][np][units]) exchange buffer: units of three
                                       // words and a tag
    int32_t polls = RES_POLLS;         // most polls of one wait
};
// 16-byte units of one cell in the exchange buffer (FP64: two per direction pair)
constexpr int resident_units(size_t state_bytes) { return state_bytes == 72 ? 8 : (int)(state_bytes / 12); }
// The resident kernel's tiles.  FP32: a thread per tile and 1-ring cell, one
// tile per SM, or several of the largest (RES_TILE): as many as its registers
// and shared memory allow.  FP64: four threads per cell (a direction pair each),
// one tile per SM.
constexpr int RES_LANES_FP64 = 4;
constexpr int RES_TILE = 256, RES_TILE_FP64 = 64;
constexpr int resident_ctas(int rsize, int maxf) { return rsize == 8 ? 1 : maxf <= 4 ? 4 : 2; }
// Its shared memory: state of the local cells, face table, the geometry of the
// gradient cells (three 2-vectors per slot; with four tiles per SM it stays in
// global memory) and the state the step began with.
template <int TILE, int MAXF, int RSIZE, int CTAS> struct ResDims : TileDims<TILE, MAXF, RSIZE> {
    typedef TileDims<TILE, MAXF, RSIZE> B;
    static constexpr bool GEO_SHARED = CTAS <= 3;
    static constexpr size_t GEO_BYTES = GEO_SHARED ? (size_t)3 * 2 * RSIZE * MAXF * TILE : 0;
    static constexpr size_t BASE_BYTES = (size_t)FVLBM_Q * RSIZE * TILE;
    static constexpr size_t BYTES = B::BYTES + GEO_BYTES + BASE_BYTES;
};

constexpr int RED_PARTS = 4;   // blocks per chunk of a reduction

enum Strategy { STRATEGY_TWO_KERNEL = 0, STRATEGY_TILE = 1 };

// Kernel launchers (fvlbm_kernels.cu).  prec = fvlbm_precision.
int launch_init_eq(const DevView& v, int prec, void* stream);
// ev: null, or 3 cudaEvent_t recorded before the face-value kernel, between
// the two kernels and after the update kernel.
int launch_stage(const DevView& v, int prec, void* stream, const void* fin, const void* fbase,
                 void* fout, double beta, int mode, void* const* ev = nullptr);
// Most kernels launched by one stage (two-kernel strategy).
constexpr int STAGE_KERNELS = 2;
inline int stage_kernels(const DevView& v) { return v.strategy == STRATEGY_TILE ? 1 : 2; }
// One translation unit per state precision.
int stage_fp64(const DevView& v, void* stream, const void* fin, const void* fbase, void* fout, double beta, int mode,
               void* const* ev);
int stage_fp32(const DevView& v, void* stream, const void* fin, const void* fbase, void* fout, double beta, int mode,
               void* const* ev);
int stage_fp16(const DevView& v, void* stream, const void* fin, const void* fbase, void* fout, double beta, int mode,
               void* const* ev);
int stage_bf16(const DevView& v, void* stream, const void* fin, const void* fbase, void* fout, double beta, int mode,
               void* const* ev);
// Resident stage loop: `stages` >= 2 stages of the scheme on state fa, with
// tags epoch + 1 .. epoch + stages - 1, none of them used before; FVLBM_ERR_UNSUPPORTED:
// not launched, the stream's part of the GPU does not hold every tile's CTA.
// resident_max_ctas: how many the whole GPU holds.
int launch_resident(const DevView& v, const ResView& r, int prec, void* stream, int scheme, int64_t stages,
                    uint32_t epoch, bool ab2_started);
int resident_max_ctas(const DevView& v, const ResView& r, int prec, int scheme);
#define FVLBM_RESIDENT_DECL(name)                                                                             \
    int name(const DevView& v, const ResView& r, void* stream, int scheme, int64_t stages, uint32_t epoch,    \
             bool ab2_started, int* max_ctas)
FVLBM_RESIDENT_DECL(resident_fp64);
FVLBM_RESIDENT_DECL(resident_fp32);
FVLBM_RESIDENT_DECL(resident_fp16);
FVLBM_RESIDENT_DECL(resident_bf16);
int launch_snapshot(const DevView& v, int prec, void* stream);
int launch_reduce(const DevView& v, int prec, void* stream, int what);
int load_reduce();   // loads the reduction's kernels on the current device (CUDA loads lazily)
// f and the macros in the caller's cell order, in a buffer the device
// accesses (host memory reachable by the GPU, or device memory).
int launch_get_f_ordered(const DevView& v, int prec, void* stream, double* f);
int launch_set_f_ordered(const DevView& v, int prec, void* stream, const double* f);
int launch_macros_ordered(const DevView& v, int prec, void* stream, double* rho, double* u);

// Solver internals for entry points defined outside the solver's own file.
struct SolverRef {
    const DevView* view;
    int prec;
    int device;
    void* stream;
    int32_t n_inst;
};
int solver_ref(fvlbm_solver* s, SolverRef* out);
// fvlbm_workspace_bytes; loop = false: without the resident loop's arrays (fvlbm_init then
// takes the solver to the stage kernels).
int workspace_bytes(const fvlbm_mesh* mesh, const fvlbm_params* params, int32_t n_params, bool loop, size_t* bytes);
// Stages of one time step, and stage k enqueued on the solver's stream (*out:
// the state buffer it writes); the last stage ends the step.
int solver_n_stages(const fvlbm_solver* s);
int solver_stage(fvlbm_solver* s, int k, void** out);
// Whether recorded steps can stand for enqueued ones (the kernels have run
// once, AB2 has its history), and which of two alternating buffers holds the state.
bool solver_replayable(const fvlbm_solver* s);
int solver_buffer(const fvlbm_solver* s);
void solver_set_buffer(fvlbm_solver* s, int b);
// What a stage costs a solver, in microseconds on a GB300: `turn` of the whole GPU in
// the resident loop (whose launches share the GPU as far as their tiles fit), or, by
// stage kernels, `base` of latency, which others' overlap, and `flow` of the whole GPU.
struct StageCost {
    double turn = 0, base = 0, flow = 0;
    double alone = 0;   // in the resident loop, nobody beside
    bool resident = false;
};
// A stage of several solvers in turns and in stage kernels that overlap; queues: how many
// run side by side.
struct OverlapGain {
    double turns = 0, left_base = 0, left_flow = 0, base = 0, flow = 0;
    int n = 0;
    void add(const StageCost& x);
    double in_turns() const { return turns + left_base + left_flow; }
    double overlapping(int queues) const { return base * ((n + queues - 1) / queues) + flow; }
};
StageCost solver_cost(const fvlbm_solver* s);
// Microseconds that a fresh request's first stage kernels take besides, for their graphs (0: it has them).
double solver_overlap_setup(const fvlbm_solver* s);
// Where the solver's next steps run (the results are the same): as fvlbm_step finds
// best, in the resident loop, or by stage kernels.
enum StepPath { STEP_AUTO = 0, STEP_RESIDENT = 1, STEP_STAGES = 2 };
void solver_path(fvlbm_solver* s, StepPath path);
// FP64 sums of a reduction (RED_MASS: [mass, -]; RED_RESIDUAL: [numerator,
// denominator]) per instance; synchronises.
int solver_sums(fvlbm_solver* s, int what, std::vector<double>& out);
// Halo exchange of a partitioned solve: entry e = (src part, src internal
// cell, dst part, dst internal cell) copies the stored state of one cell from
// part_state[src] to part_state[dst] (prec = fvlbm_precision of all parts).
int launch_halo_copy(int prec, void* stream, const int4* entries, int64_t n, void* const* part_state, int n_parts);
// Reads the solver's non-finite flag after synchronising its stream.
int solver_sync_check(fvlbm_solver* s);

// Stage modes of launch_stage.
enum StageMode { MODE_RK = 0, MODE_AB2_FIRST = 1, MODE_AB2 = 2 };
// Reductions of launch_reduce.
enum ReduceWhat { RED_MASS = 0, RED_RESIDUAL = 1 };

}  // namespace fvlbm

namespace fvlbm {
struct Adjacency;
}
struct fvlbm_mesh {
    fvlbm::Mesh m;
    // what the planner asks of it, formed by its first plan
    mutable std::mutex plan_mutex;
    mutable std::shared_ptr<const fvlbm::Adjacency> adjacency;
};

namespace fvlbm {
// One part of a partitioned mesh: its cells (caller numbering of the whole
// mesh) in local order -- owned cells ascending, then ring 1, then ring 2 --
// and its mesh (owned cells followed by the ghosts).
struct PartPlan {
    std::vector<int64_t> cells;
    int64_t n_owned = 0, n_ring1 = 0, n_ring2 = 0;
    fvlbm_mesh* mesh = nullptr;
};
// The cells part `src` sends to part `dst` after every stage: entry e is the
// owned cell src_local[e] of src (local numbering) and the ghost dst_local[e]
// of dst; cells[e] is its number in the whole mesh.
struct HaloMsg {
    int32_t src = -1, dst = -1;
    std::vector<int32_t> src_local, dst_local;
    std::vector<int64_t> cells;
};
}  // namespace fvlbm

struct fvlbm_partition {
    int32_t n_parts = 0;
    int64_t n_cell = 0;
    std::vector<int32_t> owner;            // [n_cell] part owning each cell
    std::vector<fvlbm::PartPlan> parts;
    std::vector<fvlbm::HaloMsg> msgs;      // ordered by (src, dst)
    ~fvlbm_partition();
};
