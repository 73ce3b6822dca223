// Internal declarations shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string>

#include "mlip.h"

namespace mlip {

constexpr int K_RADIAL = 32;   // radial channels (Section 3.2.3: k = 32)
constexpr int D_ANG = 16;      // irreducible angular components up to l = 3 (Section 3.3.2)
constexpr int N_INV = 128;     // (l_max + 1) * k invariants (Eq. 5)
constexpr int HEAD_H = 64;     // head width (Section 4.1.3)
constexpr int HEAD_L = 4;      // head hidden layers
constexpr int MAX_SPECIES = 8;
constexpr size_t head_net_size(int n_inv) {   // doubles per regression network in the caller's layout
    return (size_t)n_inv * HEAD_H + HEAD_H + (size_t)(HEAD_L - 1) * (HEAD_H * HEAD_H + HEAD_H) + HEAD_H + 1;
}
constexpr int HEAD_NET = (int)head_net_size(N_INV);

// 1 eV/(Angstrom amu) in Angstrom/fs^2
constexpr double ACC_UNIT = 1.602176634e-19 / 1.66053906660e-27 * 1e-10;

// device status word bits
enum : int {
    FLAG_NEIGHBOR_OVERFLOW = 1 << 0,
    FLAG_SKIN_EXCEEDED = 1 << 1,
    FLAG_NONFINITE = 1 << 2,
    FLAG_TABLE_RANGE = 1 << 3,
    FLAG_BOUNDS = 1 << 4,   // raised only by builds with -DMLIP_DEBUG_BOUNDS: an index left its array
};

// Range-checked build (-DMLIP_DEBUG_BOUNDS): every index that the fused kernels and the export take from a list or an
// order array, and every place and entry that lanes write to a list, is compared with its array's size before it is used; an index out of range raises FLAG_BOUNDS and is
// replaced by 0, so the access still happens inside the array.  Stands in for a memory checker on the kernels' gathers.
#ifdef MLIP_DEBUG_BOUNDS
#define MLIP_CHECK_INDEX(idx, size, status) (((unsigned long long)(idx) < (unsigned long long)(size)) ? (idx) : (atomicOr((status), FLAG_BOUNDS), 0))
#else
#define MLIP_CHECK_INDEX(idx, size, status) (idx)
#endif

// accumulator slots (double)
enum : int { ACC_ENERGY = 0, ACC_VIRIAL = 1, ACC_KINETIC = 10, ACC_COUNT = 32 };
// launch_base, one block in doubles: [0, 4) tile_counter (MAX_SPECIES ints), [4] pair_counter, [5, 15) acc_fx, [16, 16 + ACC_COUNT) acc;
// everything up to the kinetic-energy slot of acc is zero when a fused kernel starts.  There are two such blocks: an evaluation uses one
// and clears the other, which holds the totals of the evaluation before it, for the next (but see note_capture)
constexpr int LB_PAIR = 4, LB_ACC_FX = 5, LB_ACC = 16, LB_COUNT = LB_ACC + ACC_COUNT;
constexpr size_t LAUNCH_CLEAR_BYTES = sizeof(double) * (LB_ACC + ACC_KINETIC);
static_assert(MAX_SPECIES * sizeof(int) <= LB_PAIR * sizeof(double), "tile counters must fit before the pair counter");

struct CellGrid {
    int n[3];          // cells per dimension
    double inv_edge[3];
    double box[3];
    double half[3];    // 0.5 * box, the minimum-image threshold
    int n_cells;
};

// The 16-byte chunk c of row r of a species' radial tables is stored at position c ^ table_swizzle(r) (0, 3, 4, 7 for r mod 4).
__host__ __device__ constexpr int table_swizzle(int r) { return 2 * (r & 3) + (r & 1); }

// Radial table: uniform cubic B-spline per ordered species pair and channel.
struct TableDesc {
    const float *coef;   // [C*C][knots + 3][K_RADIAL], scaled by 2^table_exp, chunks permuted (table_swizzle)
    int knots;           // number of intervals
    float r_min;
    float inv_h;         // 1 / interval width
    float r_cut2;
};

}  // namespace mlip

struct mlip_ctx {
    mlip_config cfg{};
    std::string err;
    int n_sm = 0;

    // model
    uint32_t *head_w = nullptr;  // per-species head weights as the tensor-memory image (megakernel.cu)
    float *table = nullptr;      // spline coefficients
    int table_exp[mlip::MAX_SPECIES * mlip::K_RADIAL] = {0};   // fp32 tables: power-of-two exponents per (central species, channel)
    double *mass = nullptr;      // [C] dev
    double *nhc = nullptr;       // thermostat state {v_eta[3], eta[3], scale, -} (integrate.cu)
    double nhc_nf = 0, nhc_kT = 0, nhc_q1 = 0, nhc_qk = 0;   // parameters of the last NVT call
    // fp64 path (precision = 1) only
    double *head_w_d = nullptr;  // per-species head weights, row-major and transposed (megakernel_f64.cu)
    double *table_d = nullptr;   // spline coefficients in fp64
    double *force_d = nullptr;   // [N][3]
    double *e_atom_d = nullptr;  // [N]
    double table_err_value = 0, table_err_deriv = 0;
    mlip::TableDesc tab{};

    // system (internal order: by cell, then species, then caller index)
    int64_t n = 0, cap_atoms = 0;
    int64_t n_owned = 0;           // atoms that are central atoms (caller indices below it); the rest are ghosts
    mlip::CellGrid grid{};
    int64_t cap_cells = 0;
    double4 *pos4 = nullptr;       // x, y, z, species stored as a double
    double *vel = nullptr;         // [N][3]
    int32_t *user_of = nullptr;    // internal -> caller index
    float4 *force = nullptr;       // fx, fy, fz, unused
    long long *force_fx = nullptr; // [N][3] fixed-point forces, deterministic mode only
    long long *acc_fx = nullptr;   // [10] fixed-point energy and virial, deterministic mode only
    float *e_atom = nullptr;       // E_i, internal order
    float *disp = nullptr;         // [N][3] displacement since the last build
    int32_t *center_order = nullptr;  // internal indices sorted by (species, cell)
    // second set used as the source of a rebuild
    double4 *pos4_src = nullptr;
    double *vel_src = nullptr;
    int32_t *user_src = nullptr;
    // cells
    int32_t *cell_of = nullptr;    // per source atom
    int32_t *cell_count = nullptr, *cell_start = nullptr;   // [n_cells + 1]; cell_count is zero between builds
    int32_t *bin_count = nullptr, *bin_start = nullptr;                           // [C * n_cells + 1]
    int32_t *species_start = nullptr;  // dev [C + 1] (behind build_word)
    int32_t species_host[mlip::MAX_SPECIES + 1] = {0};   // its copy since the last synchronising build (rebuilds inside steps do not change it)
    // lists
    int32_t *nbr_count = nullptr;  // [N]
    int32_t *nbr_near = nullptr;   // [N] leading entries of each list that were within r_cut + skin / 2 at build time
    int *far_flag = nullptr;       // raised once an atom has moved skin / 4 since the build: the far entries count again
    int64_t *nbr_off = nullptr;    // [N + 1]
    int32_t *nbr = nullptr;        // list entries: int32 indices, or uint16 cell-relative codes when list16
    bool list16 = false;           // format of the current lists (mlip_config.list_format = 1 on a grid of >= 3 cells per edge)
    int32_t *cell_id = nullptr;    // [N] build-time cell of each atom as packed coordinates, internal order (allocated for list_format = 1)
    unsigned long long *tile_state = nullptr;   // [tile_words(N)] look-back words of the one-pass build
    int *build_word = nullptr;     // {ticket, private overflow flag, total entries (64 bits)} of the one-pass build, then status, rebuild_flag, far_flag, number of long lists (LONG_LIST), species_start
    float4 *rel_pos = nullptr;     // cell-relative positions of the build in progress
    int *build_host = nullptr;     // pinned copy, and the ticket of the report that wrote it
    int reports = 0;
    static constexpr int BUILD_WORDS = 8 + mlip::MAX_SPECIES + 1;
    int64_t nbr_cap = 0, n_entries = 0, n_long = 0;   // (entries, long lists: of the last synchronising build)
    // scratch
    int64_t *scan_tmp = nullptr;   // block sums for the scans
    int64_t scan_tmp_cap = 0;
    double *launch_base = nullptr;    // [2][LB_COUNT]: tile_counter, pair_counter, acc_fx, acc back to back, twice; the pointers are into
                                      // the block of the last evaluation
    bool captured = false;            // calls of this context have been captured into a graph (note_capture)
    double *acc = nullptr;         // [ACC_COUNT] (inside launch_base)
    double *kin_part = nullptr;    // [1184] per-block kinetic-energy sums, then the ticket of the last block (integrate.cu)
    unsigned long long *pair_counter = nullptr;
    int *status = nullptr;         // device status word
    int *rebuild_flag = nullptr;   // set when an atom has moved beyond the rebuild trigger; pinned copy in rebuild_host
    int *rebuild_host = nullptr;
    int64_t n_builds = 0;
    int lookback_spin_limit = 0;              // polls before a look-back wait of the one-pass list build gives up (0 = default)
    long long lookback_unpublished_tile = -1; // diagnostic list builds only (mlip_debug_rebuild)
    int *tile_counter = nullptr;   // [MAX_SPECIES] dynamic tile scheduler, one counter per central species
    int *status_host = nullptr;    // pinned
    int64_t *total_host = nullptr; // pinned
    double *stage_pos = nullptr;   // [N][3] staging for host entry point
    int32_t *stage_species = nullptr;
    float *stage_force = nullptr;
    double *stage_out = nullptr;   // [10]
    int64_t stage_cap = 0;

    bool built = false, forces_current = false;
    int kernel_ready = 0;          // fused kernels whose shared-memory limit this context has set, a bit each (fp64: whether)
    size_t table_bytes = 0;
    int64_t step = 0;
    int64_t launches = 0;
    size_t resident = 0;
    cudaStream_t last_stream = nullptr;
    bool lists_fresh = true;       // lists were built since the last evaluation was launched
    bool force_cleared = false;    // the forces were cleared for the next evaluation by a kernel before it
    // Timing marks: a ring of events, each the end of a timed part that began at the mark before it (consecutive parts share
    // a mark), or the beginning of one.
    static constexpr int EV_POOL = 256, MARKS = 4 * EV_POOL;
    cudaEvent_t mark_ev[MARKS] = {nullptr};
    unsigned char mark_kind[MARKS] = {0};
    cudaEvent_t check_ev = nullptr;   // the displacement trigger's answer has reached the host
    int64_t marks = 0;             // recorded so far
    int64_t mark_reset[4] = {0};   // per kind: parts that ended before this mark have been reset
    bool mark_open = false;        // nothing untimed has been enqueued since the last mark
    cudaStream_t mark_stream = nullptr;
    // Below STAMP_BELOW_ATOMS the kernels of a step write their own begin and end times instead: an event between two kernels costs
    // some 1.5 us and keeps the second from starting early.  Ring in two halves, each reset (begin all ones, end zero) on entry.
    static constexpr int STAMPS = 8 * EV_POOL;
    unsigned long long *stamp = nullptr;   // dev: begin [STAMPS], end [STAMPS], nanoseconds of the device's timer
    unsigned char stamp_kind[STAMPS] = {0};
    int64_t stamps = 0, stamp_reset[4] = {0};
};

namespace mlip {

#define MLIP_CUDA_TRY(ctx, call)                                                          \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess) {                                                          \
            (ctx)->err = std::string(#call) + ": " + cudaGetErrorString(e_);              \
            cudaGetLastError();   /* a later call's check must not meet this error again */ \
            return e_ == cudaErrorMemoryAllocation ? MLIP_ERR_OOM : MLIP_ERR_CUDA;        \
        }                                                                                 \
    } while (0)

// Timed parts of the path (mlip_get_timings).  Between mark_begin and mark_end only the part itself is enqueued.
enum : unsigned char { MARK_BEGIN = 0, MARK_BUILD = 1, MARK_KERNEL = 2, MARK_INTEGRATE = 3 };
inline void mark_record(mlip_ctx *c, unsigned char kind, cudaStream_t s) {
    const int slot = (int)(c->marks % mlip_ctx::MARKS);
    cudaEventRecord(c->mark_ev[slot], s);
    c->mark_kind[slot] = kind;
    c->marks += 1;
}
inline void mark_begin(mlip_ctx *c, cudaStream_t s) {
    if (!c->mark_open || c->mark_stream != s) mark_record(c, MARK_BEGIN, s);
}
inline void mark_end(mlip_ctx *c, unsigned char kind, cudaStream_t s) {
    mark_record(c, kind, s);
    c->mark_open = true;
    c->mark_stream = s;
}

// A timed kernel of a step: where it writes its times, or nullptr after recording a mark.  timed_end after its launch.
constexpr int64_t STAMP_BELOW_ATOMS = 100000;   // (about 0.6 ms a step: what the events cost is below 1 % from there on)
inline unsigned long long *timed_begin(mlip_ctx *c, unsigned char kind, cudaStream_t s) {
    if (c->n >= STAMP_BELOW_ATOMS) { mark_begin(c, s); return nullptr; }
    constexpr int R = mlip_ctx::STAMPS, H = R / 2;
    const int slot = (int)(c->stamps % R);
    if (slot % H == 0) {
        cudaMemsetAsync(c->stamp + slot, 0xff, sizeof(unsigned long long) * H, s);
        cudaMemsetAsync(c->stamp + R + slot, 0, sizeof(unsigned long long) * H, s);
    }
    c->stamp_kind[slot] = kind;
    c->stamps += 1;
    c->mark_stream = s;
    c->mark_open = false;
    return c->stamp + slot;
}
inline void timed_end(mlip_ctx *c, unsigned char kind, cudaStream_t s) { if (c->n >= STAMP_BELOW_ATOMS) mark_end(c, kind, s); }
__device__ __forceinline__ unsigned long long device_time() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void stamp_begin(unsigned long long *stamp) { if (stamp && threadIdx.x == 0) atomicMin(stamp, device_time()); }
__device__ __forceinline__ void stamp_end(unsigned long long *stamp) { if (stamp && threadIdx.x == 0) atomicMax(stamp + mlip_ctx::STAMPS, device_time()); }

// Programmatic dependent launch: a kernel launched with launch_after may start while the kernel before it on the stream is running
// (once that one's blocks have all called allow_next or ended) and calls wait_previous before it touches anything an earlier
// kernel of the stream writes or reads.  Every kernel launched this way waits in all its threads, so that "the previous kernel is
// complete" holds back along the chain.  Loads of what such kernels exchange must not be marked read-only (const __restrict__, __ldg): the
// compiler may move those across the wait.
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... A>
inline cudaError_t launch_after_if(bool early, void (*kernel)(P...), unsigned blocks, unsigned threads, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch_after(void (*kernel)(P...), unsigned blocks, unsigned threads, size_t smem, cudaStream_t s, A... args) {
    return launch_after_if(true, kernel, blocks, threads, smem, s, args...);
}

// A captured call may be replayed at any time, in any order with others: what this context remembers on the host of the launches before a
// call (which of the two blocks is clear, whether the forces are, the species' starts) then says nothing about the device.  From the
// first captured call on every evaluation keeps to one block and clears it and the forces itself, and reads the species' starts from
// the device.  Called on entry by what enqueues on a stream.
inline void note_capture(mlip_ctx *c, cudaStream_t s) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &status) != cudaSuccess) cudaGetLastError();
    if (status != cudaStreamCaptureStatusNone) c->captured = true;
}
// The two blocks of the evaluation about to be launched: its own, and the one that it clears.  set_eval_block once it is launched.
struct EvalBlocks { double *use, *clear; };
inline EvalBlocks next_eval_blocks(const mlip_ctx *c) {
    double *now = c->acc - LB_ACC, *other = now == c->launch_base ? now + LB_COUNT : c->launch_base;
    return c->captured ? EvalBlocks{now, other} : EvalBlocks{other, now};
}
inline void set_eval_block(mlip_ctx *c, double *b) {
    c->tile_counter = reinterpret_cast<int *>(b);
    c->pair_counter = reinterpret_cast<unsigned long long *>(b + LB_PAIR);
    c->acc_fx = reinterpret_cast<long long *>(b + LB_ACC_FX);
    c->acc = b + LB_ACC;
}

struct EvalClear {
    float4 *force;       // nullptr: not accumulated into (deterministic mode, fp64 contexts)
    double *force_d;     // fp64 contexts
};
EvalClear eval_clear(mlip_ctx *c);   // integrate.cu

// neighbor.cu
int launch_build(mlip_ctx *c, bool allow_sync_grow, const double *pos, const int32_t *species, cudaStream_t s);
int64_t tile_words(int64_t n);
int launch_export(mlip_ctx *c, int64_t *seg_ptr, int32_t *nbr, int64_t capacity, int64_t *n_entries_host, cudaStream_t s);
int launch_export_noalloc(mlip_ctx *c, int64_t *seg_ptr, int32_t *nbr, int64_t capacity, int64_t *n_entries_host, cudaStream_t s);
// tables.cu
int build_tables(mlip_ctx *c, const double *enc_w_host, size_t n_enc);
// megakernel.cu
int upload_head(mlip_ctx *c, const double *head_w_host);
int launch_megakernel(mlip_ctx *c, cudaStream_t s);
// megakernel_f64.cu
int upload_head_f64(mlip_ctx *c, const double *head_w_host);
int launch_megakernel_f64(mlip_ctx *c, cudaStream_t s);
bool f64_shape_supported(int k, int l_max, int basis);
// integrate.cu
int launch_kick_drift(mlip_ctx *c, double dt, bool close_step, cudaStream_t s, const double *vscale = nullptr);
int launch_scale_velocities(mlip_ctx *c, cudaStream_t s);
int launch_kick(mlip_ctx *c, double dt, cudaStream_t s);
int launch_nvt_between(mlip_ctx *c, double dt, cudaStream_t s);
int launch_kinetic(mlip_ctx *c, int change, bool thermostat, double dt, cudaStream_t s);
int launch_outputs(mlip_ctx *c, float *forces, float *e_atom, double *energy, double *virial, cudaStream_t s);
int launch_outputs_f64(mlip_ctx *c, double *forces, double *e_atom, double *energy, double *virial, cudaStream_t s);
int launch_set_positions(mlip_ctx *c, const double *pos, cudaStream_t s);
int launch_set_velocities(mlip_ctx *c, const double *vel, cudaStream_t s);
int launch_get_state(mlip_ctx *c, double *pos, double *vel, cudaStream_t s);

// Compact list entries (neighbor.cu): cell number in the 27-cell traversal order << L16_SHIFT | position inside that cell.
constexpr int L16_SHIFT = 11, L16_MASK = (1 << L16_SHIFT) - 1;
// cell_id[] holds an atom's build-time cell as packed coordinates (10 bits each: no division on the way to the 27 cell
// bases an atom's list needs); grids with more than 1,024 cells along a dimension keep int32 lists.
constexpr int CELL_PACK_BITS = 10, CELL_PACK_MAX = 1 << CELL_PACK_BITS;
__host__ __device__ inline int pack_cell(const CellGrid &g, int linear) {
    const int cz = linear % g.n[2], cy = (linear / g.n[2]) % g.n[1], cx = linear / (g.n[2] * g.n[1]);
    return cx | (cy << CELL_PACK_BITS) | (cz << (2 * CELL_PACK_BITS));
}
__host__ __device__ inline int neighbor_cell(const CellGrid &g, int cid, int it) {
    const int cx = cid & (CELL_PACK_MAX - 1), cy = (cid >> CELL_PACK_BITS) & (CELL_PACK_MAX - 1), cz = cid >> (2 * CELL_PACK_BITS);
    int x = cx + it / 9 - 1, y = cy + (it / 3) % 3 - 1, z = cz + it % 3 - 1;
    x = x < 0 ? x + g.n[0] : (x >= g.n[0] ? x - g.n[0] : x);
    y = y < 0 ? y + g.n[1] : (y >= g.n[1] ? y - g.n[1] : y);
    z = z < 0 ? z + g.n[2] : (z >= g.n[2] ? z - g.n[2] : z);
    return (x * g.n[1] + y) * g.n[2] + z;
}

// Exact minimum-image squared distance in fp64, every operation rounded on its own
// (no fused multiply-add), identical on host and device.
__device__ __forceinline__ double min_image(double d, double box, double half) {
    if (d > half) d = __dsub_rn(d, box);
    else if (d < -half) d = __dadd_rn(d, box);
    return d;
}

// Optional per-phase cycle counters (profiling builds only: -DMLIP_PHASE_CLOCKS).  Slots 16.. of
// the accumulator array receive the summed clock64 ticks of lane 0 of every warp.
#ifdef MLIP_PHASE_CLOCKS
struct PhaseClock {
    long long t, acc[16];
    __device__ __forceinline__ void start() { t = clock64(); for (int q = 0; q < 16; ++q) acc[q] = 0; }
    __device__ __forceinline__ void mark(int slot) { const long long now = clock64(); acc[slot] += now - t; t = now; }
    __device__ __forceinline__ void flush(double *a, int lane) { if (lane == 0) for (int q = 0; q < 16; ++q) atomicAdd(&a[16 + q], (double)acc[q]); }
};
#else
struct PhaseClock {
    __device__ __forceinline__ void start() {}
    __device__ __forceinline__ void mark(int) {}
    __device__ __forceinline__ void flush(double *, int) {}
};
#endif

}  // namespace mlip
