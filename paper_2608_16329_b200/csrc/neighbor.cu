// Cell binning and neighbor-list construction (Section 3.1.1: N(i) = atoms within a
// cutoff of atom i; the paper delegates this to the MD code's binning algorithm,
// Section 4.1.4).  Everything runs on the device:
//   cell id per atom -> counting sort into cell order (ties broken by species, then by the
//   caller's index, so the internal order is reproducible) -> per-species processing order
//   -> one traversal of the 27 surrounding cells, a warp per atom or a lane (list_form.cuh); two, count and fill, when there is no array
//   yet or it is too small.
// Small systems are bound by the number of launches and by the longest chain in one thread or warp, large ones by the
// traversal's instruction issue.
// The inclusion test is fp64 with separately rounded operations, so the set of pairs is
// identical to a plain CPU evaluation of the same expression.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <limits.h>
#include <string.h>
#include <type_traits>

#include "common.cuh"
#include "list_form.cuh"
#include "scan.cuh"

namespace mlip {

__device__ __forceinline__ int cell_coord(double x, double inv_edge, int n) {
    int c = (int)floor(x * inv_edge);
    return c < 0 ? 0 : (c >= n ? n - 1 : c);
}

// ---- compact list format ----
// With atoms stored in cell order a neighbor j of atom i lies in one of the 27 cells around i's cell, so an entry can
// be coded in 16 bits: the cell's number in the traversal order (0..26: x, y, z offsets ascending) in the top 5 bits, j's
// position inside that cell in the low 11 (a cell holds at most MAX_CELL_ATOMS = 1,024 atoms).  Decoding needs the build-time
// cell of i (cell_id) and the cell starts.  Half the bytes of the int32 list, the bulk of the resident footprint.
// Used when mlip_config.list_format = 1 and every dimension has at least three cells.
// One list entry in the format of the output array: the index itself, or its 16-bit code.
template <typename OUT>
__device__ __forceinline__ OUT list_entry(int j, int it, int cell_beg) {
    if (sizeof(OUT) == 2) return (OUT)((it << L16_SHIFT) | (j - cell_beg));
    return (OUT)j;
}

constexpr int LONG_WORD = 7;   // of build_word: lists with more than LONG_LIST near entries
// What a build clears on its way: the look-back words, {ticket, overflow, total} and the long lists of the one-pass traversal, and the two flags.
struct BuildClear {
    unsigned long long *tile_state;
    int64_t n_words;       // <= number of atoms
    int *build_word, *far_flag, *rebuild_flag;
};
// Cell of every atom and its rank of arrival there (cell_count is zero between builds: k_sort_gather clears it).  PACK: the atoms come
// from the caller's arrays and are packed into the source set on the way.
template <bool PACK>
__global__ void k_cell_id(const double *__restrict__ pos, const int32_t *__restrict__ species, int n_species, double4 *__restrict__ pos4,
                          int32_t *__restrict__ user, int64_t n, CellGrid g, int32_t *__restrict__ cell_of, int32_t *__restrict__ rank_of,
                          int32_t *__restrict__ cell_count, int *status, BuildClear clear) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (i < clear.n_words) clear.tile_state[i] = 0;
    if (i == 0) {
        for (int q = 0; q < 4; ++q) clear.build_word[q] = 0;
        clear.build_word[LONG_WORD] = 0;
        *clear.far_flag = 0; *clear.rebuild_flag = 0;
    }
    double4 p;
    if (PACK) {
        int s = species[i];
        if (s < 0 || s >= n_species) { atomicOr(status, FLAG_NONFINITE); s = 0; }
        p = make_double4(pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], (double)s);
        pos4[i] = p;
        user[i] = (int32_t)i;
    } else p = pos4[i];
    bool ok = (p.x >= 0.0 && p.x < g.box[0]) && (p.y >= 0.0 && p.y < g.box[1]) && (p.z >= 0.0 && p.z < g.box[2]);
    if (!ok) atomicOr(status, FLAG_NONFINITE);
    int cx = ok ? cell_coord(p.x, g.inv_edge[0], g.n[0]) : 0;
    int cy = ok ? cell_coord(p.y, g.inv_edge[1], g.n[1]) : 0;
    int cz = ok ? cell_coord(p.z, g.inv_edge[2], g.n[2]) : 0;
    int c = (cx * g.n[1] + cy) * g.n[2] + cz;
    cell_of[i] = c;
    rank_of[i] = atomicAdd(&cell_count[c], 1);
}

__global__ void k_place(const int32_t *__restrict__ cell_of, int64_t n, const int32_t *__restrict__ cell_start,
                        const int32_t *__restrict__ rank_of, int32_t *__restrict__ slot_src) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    slot_src[cell_start[cell_of[i]] + rank_of[i]] = (int32_t)i;
}

// One warp per cell: order the cell's atoms by (species, caller index) -- an atom's place is the number of smaller keys, counted in
// shared memory -- move them there from the source set (with their fp32 position relative to the cell's lower corner when `rel` is
// given: |x_rel| < cell edge, so the rounding is ~5e-7 Angstrom whatever the box size), and count the cell's central atoms per
// species (caller indices below n_owned; the others are ghosts).  One thread per cell with an insertion sort in global memory
// took 60 to 80 us at any size below 100,000 atoms, and the moves were a pass of their own.
// A cell holding more than MAX_CELL_ATOMS atoms (a collapsed or diverged configuration: thousands of atoms in a cube of
// one list radius) is not sorted and raises FLAG_NONFINITE, which makes the list kernels and the fused kernels that follow
// return at once.
constexpr int MAX_CELL_ATOMS = 1024;
constexpr int SORT_WARPS = 4;
__global__ void __launch_bounds__(SORT_WARPS * 32) k_sort_gather(CellGrid g, int n_species, const int32_t *__restrict__ cell_start,
                                                                 const int32_t *__restrict__ slot_src, const double4 *__restrict__ pos4_src,
                                                                 const double *__restrict__ vel_src, const int32_t *__restrict__ user_src,
                                                                 int32_t n_owned, double4 *__restrict__ pos4, double *__restrict__ vel,
                                                                 int32_t *__restrict__ user_of, float *__restrict__ disp, float4 *__restrict__ rel,
                                                                 int32_t *__restrict__ cell_id, int32_t *__restrict__ cell_count,
                                                                 int32_t *__restrict__ bin_count, int *status, EvalClear clear) {
    __shared__ __align__(16) int32_t s_keys[SORT_WARPS][MAX_CELL_ATOMS];
    const int lane = threadIdx.x & 31, c = blockIdx.x * SORT_WARPS + (threadIdx.x >> 5);
    if (c >= g.n_cells) return;
    int32_t *keys = s_keys[threadIdx.x >> 5];
    const int beg = cell_start[c], m = cell_start[c + 1] - beg;
    const bool sorted = m <= MAX_CELL_ATOMS;
    if (lane == 0) {
        cell_count[c] = 0;
        if (!sorted) atomicOr(status, FLAG_NONFINITE);
    }
    const int cz = c % g.n[2], cy = (c / g.n[2]) % g.n[1], cx = c / (g.n[2] * g.n[1]);
    const double corner[3] = {(double)cx * (g.box[0] / g.n[0]), (double)cy * (g.box[1] / g.n[1]), (double)cz * (g.box[2] / g.n[2])};
    const int packed = pack_cell(g, c);
    if (sorted) {
        for (int a = lane; a < ((m + 3) & ~3); a += 32) {
            int key = 0x7fffffff;
            if (a < m) { const int src = slot_src[beg + a]; key = ((int)pos4_src[src].w << 28) | user_src[src]; }
            keys[a] = key;
        }
        __syncwarp();
    }
    int owned = 0;   // lane s: central atoms of species s
    for (int base = 0; base < m; base += 32) {
        const int a = base + lane;
        int sa = -1;
        if (a < m) {
            const int src = slot_src[beg + a];
            const double4 p = pos4_src[src];
            const int user = user_src[src];
            int dst = beg + a;
            if (sorted) {
                const int key = ((int)p.w << 28) | user;
                int rank = 0;
                for (int q = 0; q < m; q += 4) {
                    const int4 o = *reinterpret_cast<const int4 *>(keys + q);
                    rank += (o.x < key) + (o.y < key) + (o.z < key) + (o.w < key);
                }
                dst = beg + rank;
            }
            pos4[dst] = p;
            user_of[dst] = user;
            if (cell_id) cell_id[dst] = packed;   // build-time cell in the internal order (compact lists)
            if (rel) rel[dst] = make_float4((float)(p.x - corner[0]), (float)(p.y - corner[1]), (float)(p.z - corner[2]), 0.f);
            for (int q = 0; q < 3; ++q) {
                vel[3 * (int64_t)dst + q] = vel_src ? vel_src[3 * (int64_t)src + q] : 0.0;
                disp[3 * (int64_t)dst + q] = 0.f;
            }
            if (clear.force) clear.force[dst] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (clear.force_d) for (int q = 0; q < 3; ++q) clear.force_d[3 * (int64_t)dst + q] = 0.0;
            if (user < n_owned) sa = (int)p.w;
        }
        for (int s = 0; s < n_species; ++s) {
            const int v = __popc(__ballot_sync(0xffffffffu, sa == s));
            if (lane == s) owned += v;
        }
    }
    if (lane < n_species) bin_count[(int64_t)lane * g.n_cells + c] = owned;
}

// One warp per cell: the cell's atoms, already species-ordered, go to their (species, cell) bins; ghosts, which come last within
// a species, are never central atoms.
__global__ void __launch_bounds__(128) k_center_order(int n_cells, int n_species, const int32_t *__restrict__ cell_start,
                                                      const double4 *__restrict__ pos4, const int32_t *__restrict__ bin_start,
                                                      int32_t *__restrict__ center_order, int32_t *__restrict__ species_start,
                                                      const int32_t *__restrict__ user_of, int32_t n_owned) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, c = tid >> 5, lane = tid & 31;
    if (tid <= n_species) species_start[tid] = bin_start[(int64_t)tid * n_cells];
    if (c >= n_cells) return;
    const int beg = cell_start[c], end = cell_start[c + 1];
    int last = -1, run = 0;   // species of the atom before this chunk and the length of its run so far
    for (int base = beg; base < end; base += 32) {
        const int a = base + lane;
        const int s = a < end ? (int)pos4[a].w : MAX_SPECIES;
        const unsigned same = __match_any_sync(0xffffffffu, s);
        const int r = __popc(same & ((1u << lane) - 1u)) + (s == last ? run : 0);
        if (a < end && user_of[a] < n_owned) center_order[bin_start[(int64_t)s * n_cells + c] + r] = a;
        last = __shfl_sync(0xffffffffu, s, 31);
        run = __shfl_sync(0xffffffffu, r, 31) + 1;
    }
}

// ---- the whole binning of a small system by one block ----
// Cell ids, counting sort, order within the cells, per-species processing order: what the kernels above do in six launches (some 35 us,
// of which the work is a third) with the per-cell state in shared memory.  An atom's place in its cell is the number of smaller keys there;
// among those of its own species it is its place in the (species, cell) bin.  An over-full cell is sorted all the same
// (the system is small) and raises the flag.  Whole synchronising build in us, six launches / one block: 256 atoms 55 / 39, 864 64 / 50,
// 2,048 66 / 58; with up to eight atoms per thread 4,000 atoms 69 / 79 and 6,912 87 / 116: one SM's memory rate, hence the limit.
constexpr int SMALL_THREADS = 1024, SMALL_PER_THREAD = 2, SMALL_ATOMS = 2048, SMALL_CELLS = 4096, SMALL_BINS = 16384;
static_assert(SMALL_ATOMS <= SMALL_THREADS * SMALL_PER_THREAD, "atoms are kept in registers");
// exclusive scan of v[0 .. n) in place, v[n] = total
__device__ __forceinline__ void small_scan(int *v, int n, int64_t *ws) {
    int carry = 0;
    for (int base = 0; base < n; base += SMALL_THREADS) {
        const int i = base + threadIdx.x;
        const int x = i < n ? v[i] : 0;
        int64_t total;
        const int ex = (int)block_exclusive_scan(x, total, ws);   // (ends with a barrier)
        if (i < n) v[i] = carry + ex;
        carry += (int)total;
    }
    if (threadIdx.x == 0) v[n] = carry;
    __syncthreads();
}
template <bool PACK>
__global__ void __launch_bounds__(SMALL_THREADS) k_bin_small(const double *__restrict__ pos, const int32_t *__restrict__ species, int n, int n_species,
                                                             int32_t n_owned, CellGrid g, const double4 *__restrict__ pos4_src, const double *__restrict__ vel_src,
                                                             const int32_t *__restrict__ user_src, double4 *__restrict__ pos4, double *__restrict__ vel,
                                                             int32_t *__restrict__ user_of, float *__restrict__ disp, float4 *__restrict__ rel,
                                                             int32_t *__restrict__ cell_id, int32_t *__restrict__ cell_start, int32_t *__restrict__ center_order,
                                                             int32_t *__restrict__ species_start, int *status, BuildClear clear, EvalClear clear_force) {
    extern __shared__ int s_small[];   // cell starts [n_cells + 1], bins [n_species * n_cells + 1], keys [n]
    __shared__ int64_t ws[33];
    int *start = s_small, *bins = start + g.n_cells + 1, *keys = bins + n_species * g.n_cells + 1;
    const int n_bins = n_species * g.n_cells;
    for (int q = threadIdx.x; q < g.n_cells + 1 + n_bins + 1; q += SMALL_THREADS) s_small[q] = 0;
    for (int q = threadIdx.x; q < clear.n_words; q += SMALL_THREADS) clear.tile_state[q] = 0;
    if (threadIdx.x == 0) {
        for (int q = 0; q < 4; ++q) clear.build_word[q] = 0;
        clear.build_word[LONG_WORD] = 0;
        *clear.far_flag = 0; *clear.rebuild_flag = 0;
    }
    __syncthreads();
    double4 p[SMALL_PER_THREAD];
    int cell[SMALL_PER_THREAD], key[SMALL_PER_THREAD], place[SMALL_PER_THREAD];
#pragma unroll
    for (int q = 0; q < SMALL_PER_THREAD; ++q) {
        const int i = threadIdx.x + q * SMALL_THREADS;
        if (i >= n) continue;
        if (PACK) {
            int s = species[i];
            if (s < 0 || s >= n_species) { atomicOr(status, FLAG_NONFINITE); s = 0; }
            p[q] = make_double4(pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], (double)s);
        } else p[q] = pos4_src[i];
        const bool ok = (p[q].x >= 0.0 && p[q].x < g.box[0]) && (p[q].y >= 0.0 && p[q].y < g.box[1]) && (p[q].z >= 0.0 && p[q].z < g.box[2]);
        if (!ok) atomicOr(status, FLAG_NONFINITE);
        const int cx = ok ? cell_coord(p[q].x, g.inv_edge[0], g.n[0]) : 0;
        const int cy = ok ? cell_coord(p[q].y, g.inv_edge[1], g.n[1]) : 0;
        const int cz = ok ? cell_coord(p[q].z, g.inv_edge[2], g.n[2]) : 0;
        cell[q] = (cx * g.n[1] + cy) * g.n[2] + cz;
        key[q] = ((int)p[q].w << 28) | (PACK ? i : user_src[i]);
        place[q] = atomicAdd(&start[cell[q]], 1);
        if ((key[q] & 0x0fffffff) < n_owned) atomicAdd(&bins[(int)p[q].w * g.n_cells + cell[q]], 1);
    }
    __syncthreads();
    small_scan(start, g.n_cells, ws);
    small_scan(bins, n_bins, ws);
    for (int q = threadIdx.x; q <= g.n_cells; q += SMALL_THREADS) cell_start[q] = start[q];
    if (threadIdx.x <= n_species) species_start[threadIdx.x] = bins[threadIdx.x * g.n_cells];
#pragma unroll
    for (int q = 0; q < SMALL_PER_THREAD; ++q)
        if (threadIdx.x + q * SMALL_THREADS < n) keys[start[cell[q]] + place[q]] = key[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < SMALL_PER_THREAD; ++q) {
        const int i = threadIdx.x + q * SMALL_THREADS;
        if (i >= n) continue;
        const int beg = start[cell[q]], end = start[cell[q] + 1], own_species = key[q] & ~0x0fffffff;
        if (end - beg > MAX_CELL_ATOMS) atomicOr(status, FLAG_NONFINITE);
        int below = 0, same = 0;   // smaller keys in the cell; those of the same species
        for (int a = beg; a < end; ++a) {
            const int o = keys[a];
            below += o < key[q];
            same += o < key[q] && o >= own_species;
        }
        const int dst = beg + below, user = key[q] & 0x0fffffff, cz = cell[q] % g.n[2], cy = (cell[q] / g.n[2]) % g.n[1], cx = cell[q] / (g.n[2] * g.n[1]);
        if (user < n_owned) center_order[bins[(int)p[q].w * g.n_cells + cell[q]] + same] = dst;
        pos4[dst] = p[q];
        user_of[dst] = user;
        if (cell_id) cell_id[dst] = pack_cell(g, cell[q]);
        if (rel) rel[dst] = make_float4((float)(p[q].x - (double)cx * (g.box[0] / g.n[0])), (float)(p[q].y - (double)cy * (g.box[1] / g.n[1])),
                                        (float)(p[q].z - (double)cz * (g.box[2] / g.n[2])), 0.f);
        for (int a = 0; a < 3; ++a) {
            vel[3 * dst + a] = vel_src ? vel_src[3 * i + a] : 0.0;
            disp[3 * dst + a] = 0.f;
        }
        if (clear_force.force) clear_force.force[dst] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (clear_force.force_d) for (int a = 0; a < 3; ++a) clear_force.force_d[3 * dst + a] = 0.0;
    }
}

// Warp per atom over the surrounding cells.  FILL = false counts, FILL = true writes the list.
// Lanes 0..26 fetch the atom ranges of the (up to) 27 cells in one round trip; the cells are then visited
// in a fixed order (x, y, z offsets ascending: the order of the list) with the positions of the next
// cell requested before the current one is tested, so that an atom costs a few load latencies instead of 54.
template <bool FILL>
__global__ void __launch_bounds__(256) k_neighbors(int64_t n, CellGrid g, double rl2, const double4 *__restrict__ pos4,
                                                   const int32_t *__restrict__ cell_start, int32_t *__restrict__ nbr_count,
                                                   const int64_t *__restrict__ nbr_off, int32_t *__restrict__ nbr,
                                                   int64_t nbr_cap, int *status, float near2, int32_t *__restrict__ nbr_near,
                                                   const int32_t *__restrict__ user_of, int32_t n_owned) {
    const int lane = threadIdx.x & 31;
    int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n || (*status & FLAG_NONFINITE)) return;   // a broken configuration is not traversed (see k_sort_gather)
    if (user_of[i] >= n_owned) {   // a ghost is listed by others but has no list of its own
        if (!FILL && lane == 0) { nbr_count[i] = 0; nbr_near[i] = 0; }
        return;
    }
    const double4 pi = pos4[i];
    // this lane's cell: offsets (ox, oy, oz) = (lane / 9, lane / 3 % 3, lane % 3); dimensions with fewer than
    // three cells list each cell once
    int cb = 0, ce = 0;
    {
        const int o[3] = {lane / 9, (lane / 3) % 3, lane % 3};
        const double p[3] = {pi.x, pi.y, pi.z};
        int cc[3];
        bool ok = lane < 27;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int na = g.n[a];
            const int c0 = cell_coord(p[a], g.inv_edge[a], na);
            int c = c0 + o[a] - 1;
            c = c < 0 ? c + na : (c >= na ? c - na : c);
            if (na < 3) { c = o[a]; ok = ok && o[a] < na; }
            cc[a] = c;
        }
        if (ok) {
            const int c = (cc[0] * g.n[1] + cc[1]) * g.n[2] + cc[2];
            cb = cell_start[c]; ce = cell_start[c + 1];
        }
    }
    const float boxf[3] = {(float)g.box[0], (float)g.box[1], (float)g.box[2]};
    const float halff[3] = {(float)g.half[0], (float)g.half[1], (float)g.half[2]};
    const float rl2_lo = (float)(rl2 * (1.0 - 1e-5)), rl2_hi = (float)(rl2 * (1.0 + 1e-5));
    int64_t off = 0;
    bool writable = true;
    int total = 0;
    if (FILL) {
        off = nbr_off[i];
        total = (int)(nbr_off[i + 1] - off);
        writable = nbr_off[i + 1] <= nbr_cap;
        if (!writable && lane == 0) atomicOr(status, FLAG_NEIGHBOR_OVERFLOW);
    }
    int cnt = 0, cn = 0;   // hits so far, near hits so far (near hits fill the list from the front, far hits from the back)
    int beg = __shfl_sync(0xffffffffu, cb, 0), end = __shfl_sync(0xffffffffu, ce, 0);
    double4 pj_next = make_double4(0.0, 0.0, 0.0, 0.0);
    if (beg + lane < end) pj_next = pos4[beg + lane];
    for (int it = 0; it < 27; ++it) {
        const int cur_beg = beg, cur_end = end;
        double4 pj = pj_next;
        if (it + 1 < 27) {   // request the first chunk of the next cell
            beg = __shfl_sync(0xffffffffu, cb, it + 1);
            end = __shfl_sync(0xffffffffu, ce, it + 1);
            if (beg + lane < end) pj_next = pos4[beg + lane];
        }
        for (int base = cur_beg; base < cur_end; base += 32) {
            const int j = base + lane;
            if (base != cur_beg && j < cur_end) pj = pos4[j];
            bool hit = false;
            float d2f = 0.f;
            if (j < cur_end && j != i) {
                const double ex = __dsub_rn(pj.x, pi.x), ey = __dsub_rn(pj.y, pi.y), ez = __dsub_rn(pj.z, pi.z);
                // fp32 screen: the squared distance to ~1e-6 relative decides every candidate that is not within
                // 1e-5 of the list radius; only those few take the exact, individually rounded fp64 predicate
                float fx = fabsf((float)ex), fy = fabsf((float)ey), fz = fabsf((float)ez);
                fx = fx > halff[0] ? boxf[0] - fx : fx;
                fy = fy > halff[1] ? boxf[1] - fy : fy;
                fz = fz > halff[2] ? boxf[2] - fz : fz;
                d2f = fx * fx + fy * fy + fz * fz;
                if (d2f < rl2_lo) hit = true;
                else if (d2f <= rl2_hi) {
                    const double dx = min_image(ex, g.box[0], g.half[0]);
                    const double dy = min_image(ey, g.box[1], g.half[1]);
                    const double dz = min_image(ez, g.box[2], g.half[2]);
                    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
                    hit = d2 < rl2;
                }
            }
            const bool near = hit && d2f < near2;
            const unsigned m = __ballot_sync(0xffffffffu, hit), mn = __ballot_sync(0xffffffffu, near), below = (1u << lane) - 1u;
            if (FILL && hit && writable)
                nbr[off + (near ? cn + __popc(mn & below) : total - 1 - (cnt - cn + __popc(m & ~mn & below)))] = j;
            cnt += __popc(m);
            cn += __popc(mn);
        }
    }
    if (!FILL && lane == 0) { nbr_count[i] = cnt; nbr_near[i] = cn; }
}

// The same traversal for grids with at least three cells per dimension, on the cell-relative fp32 positions: the
// separation is x_rel(j) - x_rel(i) + (cell offset) * edge -- the cell offset already names the periodic image, so no
// minimum-image step and no fp64 arithmetic per candidate (see launch_build for where the positions live).  Candidates within 1e-5 of the list radius (the fp32 distance is
// good to ~1e-6) are decided by the exact fp64 predicate on the full positions, so the lists are the same bit for bit.
template <bool FILL, typename OUT>
__global__ void __launch_bounds__(256) k_neighbors_rel(int64_t n, CellGrid g, double rl2, const double4 *__restrict__ pos4,
                                                       const float4 *__restrict__ rel, const int32_t *__restrict__ cell_start,
                                                       int32_t *__restrict__ nbr_count, const int64_t *__restrict__ nbr_off,
                                                       OUT *__restrict__ nbr, int64_t nbr_cap, int *status, float near2,
                                                       int32_t *__restrict__ nbr_near, const int32_t *__restrict__ user_of, int32_t n_owned) {
    const int lane = threadIdx.x & 31;
    int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n || (*status & FLAG_NONFINITE)) return;
    if (user_of[i] >= n_owned) {
        if (!FILL && lane == 0) { nbr_count[i] = 0; nbr_near[i] = 0; }
        return;
    }
    const double4 pi = pos4[i];
    const float4 ri = rel[i];
    int cb = 0, ce = 0;
    if (lane < 27) {
        const int o[3] = {lane / 9, (lane / 3) % 3, lane % 3};
        const double p[3] = {pi.x, pi.y, pi.z};
        int cc[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int na = g.n[a];
            int c = cell_coord(p[a], g.inv_edge[a], na) + o[a] - 1;
            cc[a] = c < 0 ? c + na : (c >= na ? c - na : c);
        }
        const int c = (cc[0] * g.n[1] + cc[1]) * g.n[2] + cc[2];
        cb = cell_start[c]; ce = cell_start[c + 1];
    }
    const float edge[3] = {(float)(g.box[0] / g.n[0]), (float)(g.box[1] / g.n[1]), (float)(g.box[2] / g.n[2])};
    const float rl2_lo = (float)(rl2 * (1.0 - 1e-5)), rl2_hi = (float)(rl2 * (1.0 + 1e-5));
    int64_t off = 0;
    bool writable = true;
    int total = 0;
    if (FILL) {
        off = nbr_off[i];
        total = (int)(nbr_off[i + 1] - off);
        writable = nbr_off[i + 1] <= nbr_cap;
        if (!writable && lane == 0) atomicOr(status, FLAG_NEIGHBOR_OVERFLOW);
    }
    int cnt = 0, cn = 0;
    int beg = __shfl_sync(0xffffffffu, cb, 0), end = __shfl_sync(0xffffffffu, ce, 0);
    float4 rj_next = make_float4(0.f, 0.f, 0.f, 0.f);
    if (beg + lane < end) rj_next = rel[beg + lane];
#pragma unroll
    for (int it = 0; it < 27; ++it) {
        const int cur_beg = beg, cur_end = end;
        float4 rj = rj_next;
        if (it + 1 < 27) {   // request the first chunk of the next cell
            beg = __shfl_sync(0xffffffffu, cb, it + 1);
            end = __shfl_sync(0xffffffffu, ce, it + 1);
            if (beg + lane < end) rj_next = rel[beg + lane];
        }
        // separation = x_rel(j) + shift, shift = (cell offset) * edge - x_rel(i)
        const float sx = (float)(it / 9 - 1) * edge[0] - ri.x;
        const float sy = (float)((it / 3) % 3 - 1) * edge[1] - ri.y;
        const float sz = (float)(it % 3 - 1) * edge[2] - ri.z;
        for (int base = cur_beg; base < cur_end; base += 32) {
            const int j = base + lane;
            if (base != cur_beg && j < cur_end) rj = rel[j];
            bool hit = false;
            float d2f = 0.f;
            if (j < cur_end && j != i) {
                const float dx = rj.x + sx, dy = rj.y + sy, dz = rj.z + sz;
                d2f = dx * dx + dy * dy + dz * dz;
                if (d2f < rl2_lo) hit = true;
                else if (d2f <= rl2_hi) {
                    const double4 pj = pos4[j];
                    const double ex = min_image(__dsub_rn(pj.x, pi.x), g.box[0], g.half[0]);
                    const double ey = min_image(__dsub_rn(pj.y, pi.y), g.box[1], g.half[1]);
                    const double ez = min_image(__dsub_rn(pj.z, pi.z), g.box[2], g.half[2]);
                    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
                    hit = d2 < rl2;
                }
            }
            const bool near = hit && d2f < near2;
            const unsigned m = __ballot_sync(0xffffffffu, hit), mn = __ballot_sync(0xffffffffu, near), below = (1u << lane) - 1u;
            if (FILL && hit && writable)
                nbr[off + (near ? cn + __popc(mn & below) : total - 1 - (cnt - cn + __popc(m & ~mn & below)))] = list_entry<OUT>(j, it, cur_beg);
            cnt += __popc(m);
            cn += __popc(mn);
        }
    }
    if (!FILL && lane == 0) { nbr_count[i] = cnt; nbr_near[i] = cn; }
}

// ---- one-pass variant ----
// Count and fill in a single traversal: a CTA takes a tile of 64 consecutive atoms (8 per warp; 8 atoms, one per warp, in small
// systems, where eight traversals one after the other are the kernel's time), collects each atom's hits
// in shared memory while it counts, obtains the tile's list offset from a decoupled look-back scan over the tiles before
// it (tile aggregate / inclusive prefix published in one 64-bit word, tiles handed out by a ticket so that every
// predecessor belongs to a CTA that is already running), and then copies the lists out in full rows.  Offsets are the same exclusive prefix sums the two-pass build produces, so the lists are identical.
// Every wait is bounded: after `spin_limit` polls (OP_SPIN in production) the tile raises FLAG_NEIGHBOR_OVERFLOW, publishes
// what it has and goes on.  Offsets are clamped to the capacity and a list that crosses it is cut short, so whatever the
// outcome every [nbr_off[i], nbr_off[i+1]) lies inside the array and holds atom indices.
constexpr int OP_TILE = 64;   // largest tile: the in-tile scan handles two counts per lane of one warp
constexpr int OP_SPIN = 1 << 18;

// Offsets of a tile's lists, by one warp: exclusive sums of the counts inside the tile to `off`, the entries of all tiles before it to
// *prefix and with its own to *total.
template <int TILE_ATOMS>
__device__ __forceinline__ void tile_offsets(int64_t tile, const int *cnt, long long *off, long long *prefix_out, long long *total_out, int *status,
                                             unsigned long long *tile_state, int spin_limit, long long unpublished_tile, int lane) {
    // look-back word: flag in the top two bits (0 empty, 1 tile aggregate, 2 inclusive prefix), value below
    constexpr unsigned long long OP_AGG = 1ull << 62, OP_INC = 2ull << 62, OP_VAL = (1ull << 62) - 1;
    static_assert(TILE_ATOMS <= 64, "two counts per lane");
    const int c0 = 2 * lane < TILE_ATOMS ? cnt[2 * lane] : 0, c1 = 2 * lane < TILE_ATOMS ? cnt[2 * lane + 1] : 0;
    long long incl = c0 + c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (2 * lane < TILE_ATOMS) { off[2 * lane] = incl - c0 - c1; off[2 * lane + 1] = incl - c1; }
    const long long aggregate = __shfl_sync(0xffffffffu, incl, 31);
    volatile unsigned long long *state = tile_state;
    long long prefix = 0;
    if (tile > 0) {
        if (lane == 0 && tile != unpublished_tile) state[tile] = OP_AGG | (unsigned long long)aggregate;
        int64_t hi = tile - 1;
        int spins = 0;
        for (;;) {   // windows of 32 predecessors, nearest first
            const int64_t p = hi - lane;
            unsigned long long v = OP_INC;
            if (p >= 0) v = state[p];
            const unsigned flag = (unsigned)(v >> 62);
            const unsigned inc = __ballot_sync(0xffffffffu, flag == 2), empty = __ballot_sync(0xffffffffu, flag == 0);
            const int first_inc = inc ? __ffs(inc) - 1 : 32;
            const unsigned need = first_inc >= 31 ? 0xffffffffu : ((2u << first_inc) - 1u);
            if (empty & need) {   // a tile in the window has not published yet
                if (++spins > spin_limit) { if (lane == 0) atomicOr(status, FLAG_NEIGHBOR_OVERFLOW); break; }
                __nanosleep(200);
                continue;
            }
            long long val = (lane <= first_inc && p >= 0) ? (long long)(v & OP_VAL) : 0;
#pragma unroll
            for (int o = 16; o; o >>= 1) val += __shfl_xor_sync(0xffffffffu, val, o);
            prefix += val;
            if (first_inc < 32) break;
            hi -= 32;
        }
    }
    if (lane == 0) {
        if (tile != unpublished_tile) state[tile] = OP_INC | (unsigned long long)(prefix + aggregate);
        *prefix_out = prefix;
        *total_out = prefix + aggregate;
    }
}

__device__ __forceinline__ bool rel_hit(const float4 &rj, float sx, float sy, float sz, float rl2_lo, float rl2_hi, double rl2,
                                        const double4 &pi, const double4 *__restrict__ pos4, int j, const CellGrid &g, float &d2f) {
    const float dx = rj.x + sx, dy = rj.y + sy, dz = rj.z + sz;
    d2f = dx * dx + dy * dy + dz * dz;
    if (d2f < rl2_lo) return true;
    if (d2f > rl2_hi) return false;
    const double4 pj = pos4[j];
    const double ex = min_image(__dsub_rn(pj.x, pi.x), g.box[0], g.half[0]);
    const double ey = min_image(__dsub_rn(pj.y, pi.y), g.box[1], g.half[1]);
    const double ez = min_image(__dsub_rn(pj.z, pi.z), g.box[2], g.half[2]);
    return __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez)) < rl2;
}

// The same decision on the full positions: fp32 screen after the minimum image, exact predicate near the list radius.
__device__ __forceinline__ bool full_hit(const double4 &pj, const double4 &pi, float rl2_lo, float rl2_hi, double rl2, const CellGrid &g, float &d2f) {
    const double ex = min_image(__dsub_rn(pj.x, pi.x), g.box[0], g.half[0]);
    const double ey = min_image(__dsub_rn(pj.y, pi.y), g.box[1], g.half[1]);
    const double ez = min_image(__dsub_rn(pj.z, pi.z), g.box[2], g.half[2]);
    const float fx = (float)ex, fy = (float)ey, fz = (float)ez;
    d2f = fx * fx + fy * fy + fz * fz;
    if (d2f < rl2_lo) return true;
    if (d2f > rl2_hi) return false;
    return __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez)) < rl2;
}

// atom ranges of the 27 cells around position p, one cell per lane (lanes 27.. get an empty range); !REL: a dimension with fewer
// than three cells lists each of them once
template <bool REL>
__device__ __forceinline__ void cell_ranges(const double4 &p4, const CellGrid &g, const int32_t *__restrict__ cell_start, int lane,
                                            int &cb, int &ce) {
    cb = 0; ce = 0;
    if (lane < 27) {
        const int o[3] = {lane / 9, (lane / 3) % 3, lane % 3};
        const double p[3] = {p4.x, p4.y, p4.z};
        int cc[3];
        bool ok = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int na = g.n[a];
            int c = cell_coord(p[a], g.inv_edge[a], na) + o[a] - 1;
            cc[a] = c < 0 ? c + na : (c >= na ? c - na : c);
            if (!REL && na < 3) { cc[a] = o[a]; ok = ok && o[a] < na; }
        }
        if (!ok) return;
        const int c = (cc[0] * g.n[1] + cc[1]) * g.n[2] + cc[2];
        cb = cell_start[c]; ce = cell_start[c + 1];
    }
}

// One atom's traversal for the one-pass build.  Near hits (inside near2) go to out[0], out[1], ..., far hits to out[top],
// out[top - 1], ...; only positions below `limit` are written.  Shared-memory pass: top = capacity - 1 (if the list is
// longer than the buffer the two ends collide and the list is traversed again); global pass: top = list length - 1.
// Returns the number of hits, and the number of near hits in `n_near`.
// REL = false: grids with fewer than three cells in a dimension, on the full positions with the minimum image (as k_neighbors).
template <bool REL, typename OUT, typename ENTRY>
__device__ __forceinline__ int onepass_traverse(int64_t i, const CellGrid &g, double rl2, const float (&edge)[3], float rl2_lo, float rl2_hi,
                                                const double4 *__restrict__ pos4, const float4 *__restrict__ rel,
                                                const int32_t *__restrict__ cell_start, int lane, OUT *out, int top, int limit,
                                                float near2, int &n_near) {
    // OUT = type of the buffer written here (int32 in shared memory), ENTRY = format of the list (int32 or uint16)
    const double4 pi = pos4[i];
    float4 ri = make_float4(0.f, 0.f, 0.f, 0.f);
    if (REL) ri = rel[i];
    int cb, ce;
    cell_ranges<REL>(pi, g, cell_start, lane, cb, ce);
    int cnt = 0, cn = 0;
    auto take = [&](bool hit, float d2f, int j, int it, int cell_beg) {
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (!m) return;   // (most chunks of the outer cells)
        const bool near = d2f < near2;
        const unsigned mn = __ballot_sync(0xffffffffu, hit && near), below = (1u << lane) - 1u;
        const int slot = near ? cn + __popc(mn & below) : top - (cnt - cn + __popc(m & ~mn & below));
        if (hit && slot >= 0 && slot < limit) out[slot] = (OUT)list_entry<ENTRY>(j, it, cell_beg);
        cnt += __popc(m);
        cn += __popc(mn);
    };
    if (!REL) {
        const unsigned cells = __ballot_sync(0xffffffffu, ce > cb);
        for (unsigned left = cells; left; left &= left - 1) {   // (up to 27 cells, each once)
            const int it = __ffs(left) - 1;
            const int beg = __shfl_sync(0xffffffffu, cb, it), end = __shfl_sync(0xffffffffu, ce, it);
#pragma unroll 4
            for (int base = beg; base < end; base += 32) {
                const int j = base + lane;
                float d2f = 0.f;
                const bool hit = j < end && j != i && full_hit(pos4[j < end ? j : beg], pi, rl2_lo, rl2_hi, rl2, g, d2f);
                take(hit, d2f, j, it, beg);
            }
        }
        n_near = cn;
        return cnt;
    }
    int beg = __shfl_sync(0xffffffffu, cb, 0), end = __shfl_sync(0xffffffffu, ce, 0);
    float4 rj_next = make_float4(0.f, 0.f, 0.f, 0.f);
    if (beg + lane < end) rj_next = rel[beg + lane];
#pragma unroll
    for (int it = 0; it < 27; ++it) {
        const int cur_beg = beg, cur_end = end;
        float4 rj = rj_next;
        if (it + 1 < 27) {
            beg = __shfl_sync(0xffffffffu, cb, it + 1);
            end = __shfl_sync(0xffffffffu, ce, it + 1);
            if (beg + lane < end) rj_next = rel[beg + lane];
        }
        const float sx = (float)(it / 9 - 1) * edge[0] - ri.x;
        const float sy = (float)((it / 3) % 3 - 1) * edge[1] - ri.y;
        const float sz = (float)(it % 3 - 1) * edge[2] - ri.z;
        for (int base = cur_beg; base < cur_end; base += 32) {
            const int j = base + lane;
            if (base != cur_beg && j < cur_end) rj = rel[j];
            float d2f = 0.f;
            const bool hit = j < cur_end && !(it == 13 && j == i) && rel_hit(rj, sx, sy, sz, rl2_lo, rl2_hi, rl2, pi, pos4, j, g, d2f);
            take(hit, d2f, j, it, cur_beg);
        }
    }
    n_near = cn;
    return cnt;
}

constexpr int OP_BUF = 160;   // hits kept per atom in shared memory; a longer list is traversed again straight into global memory

template <bool REL, int PER_WARP, typename ENTRY>
__global__ void __launch_bounds__(256) k_neighbors_onepass(int64_t n, CellGrid g, double rl2, const double4 *__restrict__ pos4,
                                                           const float4 *__restrict__ rel, const int32_t *__restrict__ cell_start,
                                                           int64_t *__restrict__ nbr_off, ENTRY *__restrict__ nbr, int64_t nbr_cap,
                                                           int *status, unsigned long long *tile_state, int *build_word,
                                                           const int *global_status, int spin_limit, long long unpublished_tile,
                                                           float near2, int32_t *__restrict__ nbr_near,
                                                           const int32_t *__restrict__ user_of, int32_t n_owned) {
    // `unpublished_tile` >= 0 (diagnostic builds of the lists only) names a tile that never publishes its look-back word,
    // so that its successor's bounded wait can be seen to run out; -1 in production.
    if (*global_status & FLAG_NONFINITE) return;   // a broken configuration is not traversed (see k_sort_gather)
    constexpr int TILE_ATOMS = 8 * PER_WARP;
    extern __shared__ int32_t s_hits[];   // [TILE_ATOMS][OP_BUF]
    __shared__ int s_cnt[OP_TILE], s_near[OP_TILE];
    __shared__ long long s_off[OP_TILE];
    __shared__ long long s_prefix, s_total;
    __shared__ int s_tile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_tile = atomicAdd(build_word, 1);
    __syncthreads();
    const int64_t tile = s_tile, first = tile * TILE_ATOMS;
    const float edge[3] = {(float)(g.box[0] / g.n[0]), (float)(g.box[1] / g.n[1]), (float)(g.box[2] / g.n[2])};
    const float rl2_lo = (float)(rl2 * (1.0 - 1e-5)), rl2_hi = (float)(rl2 * (1.0 + 1e-5));

    // ---- traversal: count, keep the hits ----
    for (int a = 0; a < PER_WARP; ++a) {
        const int slot = warp * PER_WARP + a;
        const int64_t i = first + slot;
        int cnt = 0, cn = 0;
        if (i < n && user_of[i] < n_owned)   // (a ghost has no list of its own)
            cnt = onepass_traverse<REL, int32_t, ENTRY>(i, g, rl2, edge, rl2_lo, rl2_hi, pos4, rel, cell_start, lane, s_hits + slot * OP_BUF, OP_BUF - 1, OP_BUF, near2, cn);
        if (lane == 0) { s_cnt[slot] = cnt; s_near[slot] = cn; }
    }
    __syncthreads();

    // ---- offsets: scan inside the tile, look back over the tiles before it ----
    if (warp == 0) tile_offsets<TILE_ATOMS>(tile, s_cnt, s_off, &s_prefix, &s_total, status, tile_state, spin_limit, unpublished_tile, lane);
    if (warp == 1) {
        unsigned longer = __popc(__ballot_sync(0xffffffffu, lane < TILE_ATOMS && s_near[lane] > LONG_LIST));
        if (TILE_ATOMS > 32) longer += __popc(__ballot_sync(0xffffffffu, s_near[(lane + 32) % OP_TILE] > LONG_LIST));
        if (lane == 0 && longer) atomicAdd(build_word + LONG_WORD, (int)longer);
    }
    __syncthreads();
    const long long tile_off = s_prefix;
    if (first + TILE_ATOMS >= n && threadIdx.x == 0) {   // the last tile closes the offsets
        nbr_off[n] = s_total < nbr_cap ? s_total : nbr_cap;
        *reinterpret_cast<long long *>(build_word + 2) = s_total;   // for the host: {ticket, overflow, total}
    }

    // ---- write the lists: full rows from shared memory ----
    for (int a = 0; a < PER_WARP; ++a) {
        const int slot = warp * PER_WARP + a;
        const int64_t i = first + slot;
        if (i >= n) break;
        const long long off = tile_off + s_off[slot];
        const int cnt = s_cnt[slot];
        int fit = cnt;   // entries of this list that the array still holds
        if (off + cnt > nbr_cap) {
            if (lane == 0) atomicOr(status, FLAG_NEIGHBOR_OVERFLOW);
            fit = off < nbr_cap ? (int)(nbr_cap - off) : 0;
        }
        const int near = s_near[slot];
        if (lane == 0) { nbr_off[i] = off < nbr_cap ? off : nbr_cap; nbr_near[i] = near < fit ? near : fit; }
        if (fit == 0) continue;
        if (cnt <= OP_BUF) {   // near hits sit at the front of the buffer, far hits at its back
            const int32_t *src = s_hits + slot * OP_BUF;
            for (int e = lane; e < fit; e += 32) nbr[off + e] = (ENTRY)src[e < near ? e : e + (OP_BUF - cnt)];
        } else {
            int cn;
            onepass_traverse<REL, ENTRY, ENTRY>(i, g, rl2, edge, rl2_lo, rl2_hi, pos4, rel, cell_start, lane, nbr + off, cnt - 1, fit, near2, cn);
        }
    }
}

// ---- lane = central atom ----
// The same lists from the same tiles of 64 atoms, two warps to a tile, for systems that fill the chip that way: each lane owns one of 32
// consecutive atoms, the candidates of the cells around them pass through shared memory 32 at a time and every lane tests every
// one (a broadcast read, packed fp32 arithmetic, no ballots and no ranks: a lane appends to its own row).  Consecutive atoms lie in cells that
// follow one another along z, so the cells around them are nine columns of (cells spanned + 2) layers; a lane takes part in the
// three layers around its own cell only.  Each lane meets the candidates in the order of the warp-per-atom traversal, with the same
// arithmetic, so the lists agree entry by entry.
// Rows hold 16-bit codes (near hits from the front, far hits from the back); `buf` entries, a multiple of four (list_lane_row).  A list that its row may
// not hold is counted to its end and then traversed a second time, in the same way, straight into its place in the array: systems of uneven density,
// whose lists are longer than the mean tells, cost no more than with an atom to a warp.  Whole build in us, 8 atoms to a warp / one to a lane:
// 108,000 atoms filling their box 470 / 271, half of it 472 / 390, a quarter 469 / 414; 1,000,188 in half of their box 2801 / 2212; 97,336 of
// 274-entry lists in half of theirs 1298 / 768; a ball of 123,161 in 161 Angstrom 445 / 380.  (Rows of 160 entries at least would hold more of those lists,
// 266 us for the first half-empty box, but fewer tiles fit an SM where lists are short: one species 432,000 atoms 519 / 563.)
constexpr int LN_WARPS = OP_TILE / 32, LN_THREADS = 32 * LN_WARPS;
constexpr int LN_SPAN = 4;                          // cells along z that a group of lanes may span: 9 x 6 cells, two to a lane
constexpr int LN_STAGE = 2 * 3 * 32;                // two chunks of candidates, x, y, z
static_assert(9 * (LN_SPAN + 2) <= 64, "cell ranges, two per lane");
__host__ __device__ constexpr int ln_row(int buf) { return buf + 2; }   // in entries: an odd number of words
inline size_t ln_smem(int buf) { return sizeof(float) * LN_STAGE * LN_WARPS + sizeof(uint16_t) * OP_TILE * ln_row(buf); }

__device__ __forceinline__ float2 pack_add(float2 a, float b) {
    unsigned long long ra, rb, rd;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %1};" : "=l"(rb) : "f"(b));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(ra), "l"(rb));
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(rd));
    return d;
}
__device__ __forceinline__ float2 pack_norm2(float2 x, float2 y, float2 z) {   // x x + y y + z z, rounded as fma(z, z, fma(y, y, x x))
    unsigned long long rx, ry, rz, rd;
    asm("mov.b64 %0, {%1, %2};" : "=l"(rx) : "f"(x.x), "f"(x.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(ry) : "f"(y.x), "f"(y.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rz) : "f"(z.x), "f"(z.y));
    asm("mul.rn.f32x2 %0, %1, %1;" : "=l"(rd) : "l"(rx));
    asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(rd) : "l"(ry));
    asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(rd) : "l"(rz));
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(rd));
    return d;
}

template <typename ENTRY>
__global__ void __launch_bounds__(LN_THREADS) k_neighbors_lanes(int64_t n, CellGrid g, double rl2, const double4 *__restrict__ pos4,
                                                                const float4 *__restrict__ rel, const int32_t *__restrict__ cell_start,
                                                                int64_t *__restrict__ nbr_off, ENTRY *__restrict__ nbr, int64_t nbr_cap,
                                                                int *status, unsigned long long *tile_state, int *build_word,
                                                                const int *global_status, int spin_limit, long long unpublished_tile,
                                                                float near2, int32_t *__restrict__ nbr_near,
                                                                const int32_t *__restrict__ user_of, int32_t n_owned, int buf) {
    if (*global_status & FLAG_NONFINITE) return;   // a broken configuration is not traversed (see k_sort_gather)
    extern __shared__ __align__(16) float s_lanes[];
    __shared__ int s_cnt[OP_TILE];
    __shared__ long long s_off[OP_TILE];
    __shared__ long long s_prefix, s_total;
    __shared__ int s_tile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_tile = atomicAdd(build_word, 1);
    __syncthreads();
    const int64_t tile = s_tile, first = tile * OP_TILE + 32 * warp, i = first + lane;
    float *stage = s_lanes + warp * LN_STAGE;
    uint16_t *rows = reinterpret_cast<uint16_t *>(s_lanes + LN_WARPS * LN_STAGE) + 32 * warp * ln_row(buf), *row = rows + lane * ln_row(buf);
    const float edge[3] = {(float)(g.box[0] / g.n[0]), (float)(g.box[1] / g.n[1]), (float)(g.box[2] / g.n[2])};
    const float rl2_lo = (float)(rl2 * (1.0 - 1e-5)), rl2_hi = (float)(rl2 * (1.0 + 1e-5));
    constexpr float FAR_AWAY = 1e18f;   // no hit, and no overflow in the squared distance

    // ---- traversal ----
    const bool live = i < n && user_of[i] < n_owned;   // (a ghost has no list of its own)
    float4 ri = make_float4(0.f, 0.f, 0.f, 0.f);
    int cx = 0, cy = 0, cz = 0;
    if (live) {
        const double4 p = pos4[i];
        ri = rel[i];
        cx = cell_coord(p.x, g.inv_edge[0], g.n[0]); cy = cell_coord(p.y, g.inv_edge[1], g.n[1]); cz = cell_coord(p.z, g.inv_edge[2], g.n[2]);
    }
    const float rl2_mid = (float)rl2, band = (float)(rl2 * 1.1e-5);
    // shared-memory addresses of the places for the next near and the next far hit.  Where the two might cross the lane begins its row again: from
    // there on it counts, and its list is traversed a second time.
    const int row_at = (int)__cvta_generic_to_shared(row), row_end = row_at + 2 * (buf - 1);
    int near_at = row_at, far_at = row_end, near_lost = 0, lost = 0;   // lost: hits whose places were given to others
    // second traversal: places in the list itself, of which `fit` are written
    ENTRY *list = nullptr;
    long long off = 0;   // of the list
    int near_next = 0, far_next = 0, fit = 0;
    [[maybe_unused]] int *bounds = const_cast<int *>(global_status);   // (range-checked builds only write it)
    auto traverse = [&](auto second_traversal, bool part) {
        constexpr bool SECOND = decltype(second_traversal)::value;
        for (unsigned left = __ballot_sync(0xffffffffu, part); left;) {   // groups of lanes with cells along one column
            const int lead = __ffs(left) - 1;
            const int X = __shfl_sync(0xffffffffu, cx, lead), Y = __shfl_sync(0xffffffffu, cy, lead), Z = __shfl_sync(0xffffffffu, cz, lead);
            const bool mine = (left >> lane & 1u) && cx == X && cy == Y && cz - Z < LN_SPAN;   // (atoms come in cell order: cz >= Z)
            const unsigned group = __ballot_sync(0xffffffffu, mine);
            left &= ~group;
            const int layers = __shfl_sync(0xffffffffu, cz, 31 - __clz(group)) - Z + 3, per_column = 65536 / layers + 1;
            // atom range of the q-th cell of the walk (columns in x, y order, layers Z - 1 .. upwards)
            auto range = [&](int q, int &b, int &e) {
                b = e = 0;
                if (q >= 9 * layers) return;
                const int col = q * per_column >> 16;
                int x = X + col / 3 - 1, y = Y + col % 3 - 1, z = Z + (q - col * layers) - 1;
                x = x < 0 ? x + g.n[0] : (x >= g.n[0] ? x - g.n[0] : x);
                y = y < 0 ? y + g.n[1] : (y >= g.n[1] ? y - g.n[1] : y);
                z = z < 0 ? z + g.n[2] : (z >= g.n[2] ? z - g.n[2] : z);
                const int c = (x * g.n[1] + y) * g.n[2] + z;
                b = cell_start[c]; e = cell_start[c + 1];
            };
            int beg0, end0, beg1, end1;
            range(lane, beg0, end0);
            range(lane + 32, beg1, end1);
            unsigned long long cells = __ballot_sync(0xffffffffu, end0 > beg0) | (unsigned long long)__ballot_sync(0xffffffffu, end1 > beg1) << 32;
            int q = 0, cell_beg = 0, base = 0, end = 0;   // the chunk being fetched: atoms base .. of cell q
            auto advance = [&]() {
                base += 32;
                if (base < end) return true;
                if (!cells) return false;
                q = __ffsll(cells) - 1;
                cells &= cells - 1;
                cell_beg = base = __shfl_sync(0xffffffffu, q < 32 ? beg0 : beg1, q & 31);
                end = __shfl_sync(0xffffffffu, q < 32 ? end0 : end1, q & 31);
                return true;
            };
            const float4 nobody = make_float4(FAR_AWAY, FAR_AWAY, FAR_AWAY, 0.f);
            bool more = advance();
            float4 r = more && base + lane < end ? rel[base + lane] : nobody;
            for (int parity = 0; more; parity ^= 1) {
                const int col = q * per_column >> 16, dz = Z + (q - col * layers) - 1 - cz, chunk = base, pos = base - cell_beg, m = min(32, end - base);
                float *st = stage + parity * (LN_STAGE / 2);
                st[lane] = r.x; st[32 + lane] = r.y; st[64 + lane] = r.z;
                more = advance();
                if (more) r = base + lane < end ? rel[base + lane] : nobody;
                // separation = x_rel(j) + shift, shift = (cell offset) * edge - x_rel(i)
                const bool in = mine && dz >= -1 && dz <= 1;
                const float sx = in ? __fmaf_rn((float)(col / 3 - 1), edge[0], -ri.x) : FAR_AWAY;   // (rounded alike in both traversals)
                const float sy = __fmaf_rn((float)(col % 3 - 1), edge[1], -ri.y);
                const float sz = __fmaf_rn((float)dz, edge[2], -ri.z);
                const int code = ((3 * col + dz + 1) << L16_SHIFT) + pos;
                const int self = dz == 0 ? code + (int)(i - chunk) : -1;   // (the central column) the lane's own atom
                __syncwarp();   // (the buffer before last was read before the last one's barrier)
                // the hit's code (%5) to the near (%0) or far (%1) place, which moves on; predicate h: hit
#define MLIP_APPEND " setp.lt.and.f32 nr, %2, %4, h; setp.ge.and.f32 fr, %2, %4, h; selp.u32 at, %0, %1, nr;" \
                    " @h st.shared.u16 [at], %5; @nr add.s32 %0, %0, 2; @fr sub.s32 %1, %1, 2;}"
                auto test = [&](auto own_column) {
                    constexpr bool OWN = decltype(own_column)::value;
                    for (int c0 = 0; c0 < m; c0 += 8) {   // (a chunk's places behind its last candidate are out of reach)
                        float2 d2[4];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const float4 x = *reinterpret_cast<const float4 *>(st + c0 + 4 * h), y = *reinterpret_cast<const float4 *>(st + 32 + c0 + 4 * h),
                                         z = *reinterpret_cast<const float4 *>(st + 64 + c0 + 4 * h);
                            d2[2 * h] = pack_norm2(pack_add(make_float2(x.x, x.y), sx), pack_add(make_float2(y.x, y.y), sy), pack_add(make_float2(z.x, z.y), sz));
                            d2[2 * h + 1] = pack_norm2(pack_add(make_float2(x.z, x.w), sx), pack_add(make_float2(y.z, y.w), sy), pack_add(make_float2(z.z, z.w), sz));
                        }
                        float closest = 3.0e38f;   // to the list radius
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float2 off = pack_add(d2[e], -rl2_mid);
                            closest = fminf(closest, fminf(fabsf(off.x), fabsf(off.y)));
                        }
                        if (!SECOND && far_at - near_at < 2 * 7) {
                            near_lost += (near_at - row_at) >> 1;
                            lost += ((near_at - row_at) >> 1) + ((row_end - far_at) >> 1);
                            near_at = row_at; far_at = row_end;
                        }
                        if (SECOND || __any_sync(0xffffffffu, closest <= band)) {
                            // a candidate within 1e-5 of the list radius: the exact predicate on the full positions decides
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                const float v = e & 1 ? d2[e >> 1].y : d2[e >> 1].x;
                                bool hit = v <= rl2_hi && !(OWN && code + c0 + e == self);
                                if (hit && v >= rl2_lo) {
                                    const double4 pi = pos4[i], pj = pos4[MLIP_CHECK_INDEX(chunk + c0 + e, n, bounds)];
                                    const double ex = min_image(__dsub_rn(pj.x, pi.x), g.box[0], g.half[0]);
                                    const double ey = min_image(__dsub_rn(pj.y, pi.y), g.box[1], g.half[1]);
                                    const double ez = min_image(__dsub_rn(pj.z, pi.z), g.box[2], g.half[2]);
                                    hit = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez)) < rl2;
                                }
                                const bool near = v < near2;
                                if (SECOND) {
                                    const int at = near ? near_next : far_next;
                                    if (hit && (unsigned)at < (unsigned)fit) list[MLIP_CHECK_INDEX(off + at, nbr_cap, bounds) - off] = (ENTRY)(sizeof(ENTRY) == 4 ? chunk + c0 + e : code + c0 + e);
                                    near_next += hit && near; far_next -= hit && !near;
                                } else if (hit) {
                                    asm volatile("st.shared.u16 [%0], %1;" ::"r"(near ? near_at : far_at), "r"(code + c0 + e) : "memory");
                                    if (near) near_at += 2; else far_at -= 2;
                                }
                            }
                        } else {   // no branches: few lanes have a hit, and a divergent branch costs more than the instructions it skips
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                const float v = e & 1 ? d2[e >> 1].y : d2[e >> 1].x;
                                if (OWN) asm volatile("{.reg .pred h, nr, fr; .reg .u32 at; setp.ne.s32 h, %5, %6; setp.le.and.f32 h, %2, %3, h;" MLIP_APPEND
                                                      : "+r"(near_at), "+r"(far_at) : "f"(v), "f"(rl2_hi), "f"(near2), "r"(code + c0 + e), "r"(self) : "memory");
                                else asm volatile("{.reg .pred h, nr, fr; .reg .u32 at; setp.le.f32 h, %2, %3;" MLIP_APPEND
                                                  : "+r"(near_at), "+r"(far_at) : "f"(v), "f"(rl2_hi), "f"(near2), "r"(code + c0 + e) : "memory");
                            }
                        }
                    }
                };
#undef MLIP_APPEND
                if (col == 4) test(std::true_type{});
                else test(std::false_type{});
            }
            __syncwarp();   // (the next group's first chunk may go where a lane still reads)
        }
    };
    traverse(std::false_type{}, live);
    const int cn = near_lost + ((near_at - row_at) >> 1), cnt = lost + ((near_at - row_at) >> 1) + ((row_end - far_at) >> 1);   // near hits, hits
    s_cnt[32 * warp + lane] = cnt;
    __syncthreads();
    if (warp == 0) tile_offsets<OP_TILE>(tile, s_cnt, s_off, &s_prefix, &s_total, status, tile_state, spin_limit, unpublished_tile, lane);
    __syncthreads();
    if (tile * OP_TILE + OP_TILE >= n && threadIdx.x == 0) {   // the last tile closes the offsets
        nbr_off[n] = s_total < nbr_cap ? s_total : nbr_cap;
        *reinterpret_cast<long long *>(build_word + 2) = s_total;   // for the host: {ticket, overflow, total}
    }

    // ---- write the lists: full rows from shared memory ----
    off = s_prefix + s_off[32 * warp + lane];
    fit = cnt;   // entries of this list that the array still holds
    if (i < n) {
        if (off + cnt > nbr_cap) {
            atomicOr(status, FLAG_NEIGHBOR_OVERFLOW);
            fit = off < nbr_cap ? (int)(nbr_cap - off) : 0;
        }
        nbr_off[i] = off < nbr_cap ? off : nbr_cap;
        nbr_near[i] = cn < fit ? cn : fit;
    }
    const unsigned longer = __ballot_sync(0xffffffffu, cn > LONG_LIST);
    if (lane == 0 && longer) atomicAdd(build_word + LONG_WORD, __popc(longer));
    if (__any_sync(0xffffffffu, lost > 0)) {   // lists longer than their rows, straight to their places
        list = nbr + off; far_next = cnt - 1;
        traverse(std::true_type{}, lost > 0);
        if (lost > 0) fit = 0;
    }
    int cell_of_bases = -1, bases = 0;   // lane q < 27: first atom of the q-th cell around that cell
    for (int a = 0; a < 32; ++a) {
        const int m = __shfl_sync(0xffffffffu, fit, a), all = __shfl_sync(0xffffffffu, cnt, a), near = __shfl_sync(0xffffffffu, cn, a);
        if (m == 0) continue;   // (written above; atoms beyond the last and ghosts have none either)
        const long long to = __shfl_sync(0xffffffffu, off, a);
        if (sizeof(ENTRY) == 4) {
            const int X = __shfl_sync(0xffffffffu, cx, a), Y = __shfl_sync(0xffffffffu, cy, a), Z = __shfl_sync(0xffffffffu, cz, a);
            const int cell = (X * g.n[1] + Y) * g.n[2] + Z;
            if (cell != cell_of_bases) {
                cell_of_bases = cell;
                if (lane < 27) {
                    int x = X + lane / 9 - 1, y = Y + (lane / 3) % 3 - 1, z = Z + lane % 3 - 1;
                    x = x < 0 ? x + g.n[0] : (x >= g.n[0] ? x - g.n[0] : x);
                    y = y < 0 ? y + g.n[1] : (y >= g.n[1] ? y - g.n[1] : y);
                    z = z < 0 ? z + g.n[2] : (z >= g.n[2] ? z - g.n[2] : z);
                    bases = cell_start[(x * g.n[1] + y) * g.n[2] + z];
                }
            }
        }
        const uint16_t *src = rows + a * ln_row(buf);
        for (int e0 = 0; e0 < m; e0 += 32) {
            const int e = e0 + lane, code = e < m ? src[e < near ? e : e + (buf - all)] : 0;
            int entry = code;
            if (sizeof(ENTRY) == 4) entry = __shfl_sync(0xffffffffu, bases, code >> L16_SHIFT) + (code & L16_MASK);
            if (e < m) nbr[MLIP_CHECK_INDEX(to + e, nbr_cap, bounds)] = (ENTRY)MLIP_CHECK_INDEX(entry, sizeof(ENTRY) == 4 ? n : 27ll << L16_SHIFT, bounds);
        }
    }
}

// ---- canonical export: caller's indices, species-segmented, ascending ----
// Entry e of atom i's list as an internal index, whatever the list format (cell_id = nullptr: plain indices).
struct ListView {
    const int32_t *nbr;
    const uint16_t *nbr16;
    const int32_t *cell_id, *cell_start;
    CellGrid grid;
    int64_t n, nbr_cap;   // atoms, room for entries (range-checked builds)
    int *status;
    __device__ __forceinline__ int at(int64_t i, int64_t e) const {
        e = MLIP_CHECK_INDEX(e, nbr_cap, status);
        if (!nbr16) return (int)MLIP_CHECK_INDEX(nbr[e], n, status);
        const int code = nbr16[e];
        const int j = cell_start[MLIP_CHECK_INDEX(neighbor_cell(grid, cell_id[i], code >> L16_SHIFT), grid.n_cells, status)] + (code & L16_MASK);
        return (int)MLIP_CHECK_INDEX(j, n, status);
    }
};

// An atom's place in every canonical list: species, then caller index, in one word (8 species, 2^28 atoms); the lengths of the
// lists in the caller's order.
__global__ void k_export_keys(int64_t n, const double4 *__restrict__ pos4, const int32_t *__restrict__ user_of, const int64_t *__restrict__ nbr_off,
                              int32_t *__restrict__ key, int32_t *__restrict__ len) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int user = user_of[i];
    key[i] = ((int)pos4[i].w << 28) | user;
    len[user] = (int)(nbr_off[i + 1] - nbr_off[i]);
}

// Warp per atom: entries per species, one count to a lane.  Each lane counts in 16-bit fields (a list holds at most 27 x MAX_CELL_ATOMS entries).
__device__ __forceinline__ int species_counts(const ListView &lv, const int32_t *__restrict__ key, int64_t i, int64_t beg, int64_t end, int lane) {
    static_assert(27 * MAX_CELL_ATOMS < 65536 && MAX_SPECIES == 8, "16-bit fields, two to a word");
    unsigned cnt[4] = {0, 0, 0, 0};
    for (int64_t e = beg + lane; e < end; e += 32) {
        const int s = (int)((unsigned)key[lv.at(i, e)] >> 28);
#pragma unroll
        for (int w = 0; w < 4; ++w) cnt[w] += (s >> 1) == w ? 1u << (16 * (s & 1)) : 0u;
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) cnt[w] = __reduce_add_sync(0xffffffffu, cnt[w]);
    return (int)((((lane >> 1) == 0 ? cnt[0] : (lane >> 1) == 1 ? cnt[1] : (lane >> 1) == 2 ? cnt[2] : cnt[3]) >> (16 * (lane & 1))) & 0xffffu);
}
// Segment lengths without the lists (a call whose array is too small reports those): the fill kernel finds the segments itself.
__global__ void __launch_bounds__(256) k_export_count(int64_t n, int n_species, const int64_t *__restrict__ nbr_off, ListView lv,
                                                      const int32_t *__restrict__ key, int32_t *__restrict__ seg_count) {
    const int lane = threadIdx.x & 31;
    int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;
    const int count = species_counts(lv, key, i, nbr_off[i], nbr_off[i + 1], lane);
    if (lane < n_species) seg_count[(int64_t)MLIP_CHECK_INDEX(key[i] & 0x0fffffff, n, lv.status) * n_species + lane] = count;
}

// Sort of 32 x R keys by a warp, ascending in lane * R + r: a bitonic network whose phases start with a mirrored step, so that every
// compare-exchange puts the smaller key at the lower index.
template <int R>
__device__ __forceinline__ void warp_sort(int32_t (&v)[R], int lane) {
#pragma unroll
    for (int k = 2; k <= 32 * R; k <<= 1) {
        if (k <= R) {
#pragma unroll
            for (int r = 0; r < R; ++r)
                if ((r & (k >> 1)) == 0) { const int q = r ^ (k - 1); const int lo = min(v[r], v[q]); v[q] = max(v[r], v[q]); v[r] = lo; }
        } else {
            const bool lower = (lane & (k / (2 * R))) == 0;
            int32_t o[R];
#pragma unroll
            for (int r = 0; r < R; ++r) o[r] = __shfl_xor_sync(0xffffffffu, v[R - 1 - r], k / R - 1);
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = lower ? min(v[r], o[r]) : max(v[r], o[r]);
        }
#pragma unroll
        for (int j = k >> 2; j > 0; j >>= 1) {
            if (j >= R) {
                const bool lower = (lane & (j / R)) == 0;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int32_t o = __shfl_xor_sync(0xffffffffu, v[r], j / R);
                    v[r] = lower ? min(v[r], o) : max(v[r], o);
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if ((r & j) == 0) { const int lo = min(v[r], v[r ^ j]); v[r ^ j] = max(v[r], v[r ^ j]); v[r] = lo; }
            }
        }
    }
}

// Warp per atom: the list's keys sorted in registers (four or eight to a lane; they differ within a list), turned to full rows through
// shared memory and written.  Longer lists: an entry's place is the number of smaller keys, read again from global memory.
// 108,000 atoms with 134 entries each: 2.0 ms when every pair of entries was compared through list, species and caller index, 375 us
// when keys were ranked against a copy in shared memory (some 2,000 instructions per list), 110 us sorted (about 600).
// The first segment of an atom starts at seg_ptr[its caller index * n_species], which the scan of the list lengths has written; the
// others start where the species changes in the sorted keys.  (Counted by a pass of
// their own, with a scan over all n_species times as many segments: 108,000 atoms 500 instead of 463 us for build and export.)
constexpr int EXPORT_BUF = 256;
template <int R>
__device__ __forceinline__ void export_sorted(const ListView &lv, const int32_t *__restrict__ key, int64_t i, int64_t beg, int m, int32_t *keys, int n_species,
                                              int64_t off, int64_t *__restrict__ seg, int32_t *__restrict__ out, int lane) {
    int32_t v[R];
#pragma unroll
    for (int c = 0; c < R; ++c) v[c] = 32 * c + lane < m ? key[lv.at(i, beg + 32 * c + lane)] : 0x7fffffff;
    warp_sort<R>(v, lane);
#pragma unroll
    for (int c = 0; c < R; c += 4) *reinterpret_cast<int4 *>(keys + lane * R + c) = make_int4(v[c], v[c + 1], v[c + 2], v[c + 3]);
    __syncwarp();
#pragma unroll
    for (int c = 0; c < R; ++c) {
        const int e = 32 * c + lane;
        if (e < m) out[e] = keys[e] & 0x0fffffff;
    }
    if (lane > 0 && lane < n_species) {   // lane q: the entries of species below q
        int below = 0;
#pragma unroll
        for (int step = 16 * R; step; step >>= 1)
            if (keys[below + step - 1] < lane << 28) below += step;
        if (keys[below] < lane << 28) ++below;
        seg[lane] = off + below;
    }
}
__global__ void __launch_bounds__(256) k_export_fill(int64_t n, int n_species, const int64_t *__restrict__ nbr_off, ListView lv,
                                                     const int32_t *__restrict__ key, int64_t *__restrict__ seg_ptr, int32_t *__restrict__ out) {
    __shared__ __align__(16) int32_t s_keys[8][EXPORT_BUF];
    const int lane = threadIdx.x & 31;
    int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;
    int32_t *keys = s_keys[threadIdx.x >> 5];
    const int64_t beg = nbr_off[i];
    const int m = (int)(nbr_off[i + 1] - beg);
    int64_t *seg = seg_ptr + (int64_t)MLIP_CHECK_INDEX(key[i] & 0x0fffffff, n, lv.status) * n_species;   // the species' segments of an atom follow one another
    const int64_t off = *seg;
    out += off;
    if (m <= EXPORT_BUF / 2) return export_sorted<4>(lv, key, i, beg, m, keys, n_species, off, seg, out, lane);
    if (m <= EXPORT_BUF) return export_sorted<8>(lv, key, i, beg, m, keys, n_species, off, seg, out, lane);
    const int count = species_counts(lv, key, i, beg, beg + m, lane);
    int before = 0;   // lane q: entries of the species below q
    for (int q = 0; q + 1 < n_species; ++q) { const int c = __shfl_sync(0xffffffffu, count, q); before += lane > q ? c : 0; }
    if (lane > 0 && lane < n_species) seg[lane] = off + before;
    for (int e = lane; e < m; e += 32) {
        const int32_t mine = key[lv.at(i, beg + e)];
        int rank = 0;
        for (int f = 0; f < m; ++f) rank += key[lv.at(i, beg + f)] < mine;
        out[rank] = mine & 0x0fffffff;
    }
}

static inline unsigned blocks_for(int64_t n, int per_block) { return (unsigned)((n + per_block - 1) / per_block); }

static ListView list_view(const mlip_ctx *c) {
    ListView lv;
    lv.nbr = c->nbr;
    lv.nbr16 = c->list16 ? reinterpret_cast<const uint16_t *>(c->nbr) : nullptr;
    lv.cell_id = c->cell_id; lv.cell_start = c->cell_start; lv.grid = c->grid;
    lv.n = c->n; lv.nbr_cap = c->nbr_cap; lv.status = c->status;
    return lv;
}

// What a synchronising build has to know -- {ticket, overflow, total, status} and the species' starts, neighbors in memory -- is written by
// a kernel straight to page-locked host memory, where the host watches for the ticket behind it: a copy and the wait for the stream
// leave the GPU idle for longer (256-atom screening 82 -> 77 us a configuration).  After REPORT_WATCH (a large build, or one queued behind other
// work) the host waits for the stream after all; the stream is asked now and then, so that an error ends the watch.
constexpr std::chrono::microseconds REPORT_WATCH(500);
__global__ void k_report(const int *words, volatile int *host, int ticket) {
    wait_previous();
    if (threadIdx.x < mlip_ctx::BUILD_WORDS) host[threadIdx.x] = words[threadIdx.x];
    __threadfence_system();
    __syncwarp();
    if (threadIdx.x == 0) {
        __threadfence_system();
        host[mlip_ctx::BUILD_WORDS] = ticket;
    }
}
static int read_build_words(mlip_ctx *c, cudaStream_t s) {
    c->reports = c->reports == INT_MAX ? 1 : c->reports + 1;
    const int ticket = c->reports;
    volatile int *seen = c->build_host + mlip_ctx::BUILD_WORDS;
    MLIP_CUDA_TRY(c, launch_after(k_report, 1, 32, 0, s, c->build_word, c->build_host, ticket));
    c->launches += 1;
    const auto begin = std::chrono::steady_clock::now();
    for (unsigned polls = 1; *seen != ticket; ++polls) {
        if (polls % 4096) continue;
        const cudaError_t e = cudaStreamQuery(s);
        if (e != cudaErrorNotReady) { MLIP_CUDA_TRY(c, e); break; }   // (complete: the words are there)
        if (std::chrono::steady_clock::now() - begin > REPORT_WATCH) { MLIP_CUDA_TRY(c, cudaStreamSynchronize(s)); break; }
    }
    std::atomic_thread_fence(std::memory_order_acquire);
    return MLIP_OK;
}

// Long lists after a counting pass (the single traversal counts them on its way).
__global__ void k_count_long(int64_t n, const int32_t *__restrict__ nbr_near, int *count) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int longer = __syncthreads_count(i < n && nbr_near[i] > LONG_LIST);
    if (threadIdx.x == 0 && longer) atomicAdd(count, longer);
}

// A synchronising build that met a non-finite or out-of-box position, a species out of range or an over-full cell: the
// list kernels have not run, so there is nothing to size a list from.  Reports it now and clears the flag.
static int refuse_broken_input(mlip_ctx *c, cudaStream_t s) {
    mark_end(c, MARK_BUILD, s);
    MLIP_CUDA_TRY(c, cudaMemsetAsync(c->status, 0, sizeof(int), s));
    c->err = "non-finite or out-of-box position, species out of range, or more than 1024 atoms in one cell";
    return MLIP_ERR_NONFINITE;
}

int64_t tile_words(int64_t n) { return list_tile_words(n); }
static_assert(list_form_tile(ListForm::LANES) == OP_TILE, "tiles");

static ListForm form_of(const mlip_ctx *c, bool rel) {
    if (c->lookback_unpublished_tile >= 0 || c->lookback_spin_limit > 0) return rel ? ListForm::LANES : ListForm::WARP_8;   // (diagnostics name 64-atom tiles)
    return list_form(c->n, c->grid.n_cells, rel);
}

template <bool REL, int PER_WARP, typename ENTRY>
static void launch_onepass(mlip_ctx *c, ENTRY *nbr, int *flag, double rl, float near2, cudaStream_t s) {
    const int spin = c->lookback_spin_limit > 0 ? c->lookback_spin_limit : OP_SPIN;
    const int64_t n_tiles = (c->n + 8 * PER_WARP - 1) / (8 * PER_WARP);
    k_neighbors_onepass<REL, PER_WARP, ENTRY><<<(unsigned)n_tiles, 256, sizeof(int32_t) * 8 * PER_WARP * OP_BUF, s>>>(
        c->n, c->grid, rl * rl, c->pos4, c->rel_pos, c->cell_start, c->nbr_off, nbr, c->nbr_cap, flag, c->tile_state, c->build_word, c->status, spin,
        c->lookback_unpublished_tile, near2, c->nbr_near, c->user_of, (int32_t)c->n_owned);
    c->launches += 1;
}

static int lanes_row(const mlip_ctx *c, double rl) {
    const double volume = c->grid.box[0] * c->grid.box[1] * c->grid.box[2];
    return list_lane_row(c->n, (double)c->n / volume * (4.0 / 3.0 * 3.14159265358979 * rl * rl * rl), c->n_sm);
}

template <typename ENTRY>
static int launch_lanes(mlip_ctx *c, ENTRY *nbr, int *flag, double rl, float near2, cudaStream_t s) {
    const int spin = c->lookback_spin_limit > 0 ? c->lookback_spin_limit : OP_SPIN, buf = lanes_row(c, rl);
    const size_t smem = ln_smem(buf);
    if (smem > 40000) MLIP_CUDA_TRY(c, cudaFuncSetAttribute(k_neighbors_lanes<ENTRY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ln_smem(LANE_ROW_MOST)));
    k_neighbors_lanes<ENTRY><<<(unsigned)((c->n + OP_TILE - 1) / OP_TILE), LN_THREADS, smem, s>>>(
        c->n, c->grid, rl * rl, c->pos4, c->rel_pos, c->cell_start, c->nbr_off, nbr, c->nbr_cap, flag, c->tile_state, c->build_word, c->status, spin,
        c->lookback_unpublished_tile, near2, c->nbr_near, c->user_of, (int32_t)c->n_owned, buf);
    c->launches += 1;
    return MLIP_OK;
}

// Sort the source set into cell order and build the lists.  The source is (pos4_src, vel_src, user_src), filled from the caller's
// arrays first when `pos` is given (velocities then start at zero).
int launch_build(mlip_ctx *c, bool allow_sync_grow, const double *pos, const int32_t *species, cudaStream_t s) {
    mark_begin(c, s);
    c->lists_fresh = true;
    const int64_t n = c->n;
    const CellGrid &g = c->grid;
    const int C = c->cfg.n_species;
    const double rl = c->cfg.r_cut + c->cfg.skin;
    // entries farther than r_cut + skin / 2 at build time form the back part of each list: they cannot come inside r_cut
    // before some atom has moved skin / 4, and the fused kernels skip them until then (far_flag, raised by the integrator)
    const double rn = c->cfg.r_cut + 0.5 * c->cfg.skin;
    const float near2 = c->cfg.skin > 0.0 ? (float)(rn * rn * (1.0 + 1e-5)) : 3.0e38f;
    // grids of at least 3 x 3 x 3 cells take the fp32 cell-relative traversal (positions staged by the sort)
    const bool rel = g.n[0] >= 3 && g.n[1] >= 3 && g.n[2] >= 3;
    // they live in the velocity source when that is not read (a build from the caller's arrays), else in the force array, idle during
    // a build.  Where they leave it alone the forces are cleared for the evaluation that follows.
    float4 *relpos = pos ? reinterpret_cast<float4 *>(c->vel_src) : c->force;
    EvalClear clear_forces = eval_clear(c);
    if (rel && clear_forces.force == relpos) { clear_forces.force = nullptr; c->force_cleared = false; }
    c->rel_pos = relpos;
    const ListForm form = form_of(c, rel);
    const BuildClear clear{c->tile_state, (n + list_form_tile(form) - 1) / list_form_tile(form), c->build_word, c->far_flag, c->rebuild_flag};
    const int64_t n_bins = (int64_t)C * g.n_cells;
    if (n <= SMALL_ATOMS && g.n_cells <= SMALL_CELLS && n_bins <= SMALL_BINS) {
        const size_t smem = sizeof(int) * (size_t)(g.n_cells + 1 + n_bins + 1 + n);
        auto *kernel = pos ? k_bin_small<true> : k_bin_small<false>;
        if (smem > 40000) MLIP_CUDA_TRY(c, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(int) * (SMALL_CELLS + SMALL_BINS + 2 + SMALL_ATOMS))));
        kernel<<<1, SMALL_THREADS, smem, s>>>(pos, species, (int)n, C, (int32_t)c->n_owned, g, c->pos4_src, pos ? nullptr : c->vel_src, c->user_src, c->pos4, c->vel,
                                              c->user_of, c->disp, rel ? relpos : nullptr, c->cell_id, c->cell_start, c->center_order, c->species_start,
                                              c->status, clear, clear_forces);
        c->launches += 1;
    } else {
        // scratch: overwritten further down whatever the outcome (nbr_near must not hold scratch: it bounds reads of a list that a
        // broken configuration leaves as it was)
        int32_t *rank_of = c->center_order, *slot_src = c->nbr_count;
        if (pos) k_cell_id<true><<<blocks_for(n, 256), 256, 0, s>>>(pos, species, C, c->pos4_src, c->user_src, n, g, c->cell_of, rank_of, c->cell_count, c->status, clear);
        else k_cell_id<false><<<blocks_for(n, 256), 256, 0, s>>>(nullptr, nullptr, C, c->pos4_src, c->user_src, n, g, c->cell_of, rank_of, c->cell_count, c->status, clear);
        int n_launches = exclusive_scan<int32_t, int32_t>(c->cell_count, c->cell_start, g.n_cells, c->scan_tmp, s);
        k_place<<<blocks_for(n, 256), 256, 0, s>>>(c->cell_of, n, c->cell_start, rank_of, slot_src);
        k_sort_gather<<<blocks_for(g.n_cells, SORT_WARPS), SORT_WARPS * 32, 0, s>>>(g, C, c->cell_start, slot_src, c->pos4_src, pos ? nullptr : c->vel_src, c->user_src,
                                                                                   (int32_t)c->n_owned, c->pos4, c->vel, c->user_of, c->disp, rel ? relpos : nullptr,
                                                                                   c->cell_id, c->cell_count, c->bin_count, c->status, clear_forces);
        n_launches += exclusive_scan<int32_t, int32_t>(c->bin_count, c->bin_start, (int64_t)C * g.n_cells, c->scan_tmp, s);
        k_center_order<<<blocks_for((int64_t)g.n_cells * 32, 128), 128, 0, s>>>(g.n_cells, C, c->cell_start, c->pos4, c->bin_start, c->center_order, c->species_start, c->user_of, (int32_t)c->n_owned);
        c->launches += n_launches + 4;
    }
    // entry format of this build: 16-bit cell-relative codes if asked for and the grid has 27 distinct cells around every
    // cell, else plain indices.  A change of format gives up the old array (its capacity is counted in entries).
    const bool list16 = c->cfg.list_format == 1 && rel && std::max(g.n[0], std::max(g.n[1], g.n[2])) <= CELL_PACK_MAX;
    if (list16 != c->list16 && c->nbr) {
        cudaFree(c->nbr);
        c->resident -= (c->list16 ? sizeof(uint16_t) : sizeof(int32_t)) * c->nbr_cap;
        c->nbr = nullptr; c->nbr_cap = 0;
    }
    c->list16 = list16;
    const size_t entry_bytes = list16 ? sizeof(uint16_t) : sizeof(int32_t);
    uint16_t *nbr16 = reinterpret_cast<uint16_t *>(c->nbr);
    // Single traversal whenever a list array exists: always for in-step rebuilds (capacity as it stands, overflow -> status
    // bit), and for a synchronising build as a first try whose overflow flag is private and sends it to the two-pass path.
    if (c->nbr_cap > 0) {
        int *flag = allow_sync_grow ? c->build_word + 1 : c->status;
        int rc = MLIP_OK;
        if (form == ListForm::LANES) rc = list16 ? launch_lanes(c, nbr16, flag, rl, near2, s) : launch_lanes(c, c->nbr, flag, rl, near2, s);
        else if (list16) form == ListForm::WARP_1 ? launch_onepass<true, 1, uint16_t>(c, nbr16, flag, rl, near2, s) : launch_onepass<true, 8, uint16_t>(c, nbr16, flag, rl, near2, s);
        else if (rel) form == ListForm::WARP_1 ? launch_onepass<true, 1, int32_t>(c, c->nbr, flag, rl, near2, s) : launch_onepass<true, 8, int32_t>(c, c->nbr, flag, rl, near2, s);
        else form == ListForm::WARP_1 ? launch_onepass<false, 1, int32_t>(c, c->nbr, flag, rl, near2, s) : launch_onepass<false, 8, int32_t>(c, c->nbr, flag, rl, near2, s);
        if (rc != MLIP_OK) return rc;
        MLIP_CUDA_TRY(c, cudaGetLastError());
        bool done = true;
        if (allow_sync_grow) {
            if ((rc = read_build_words(c, s)) != MLIP_OK) return rc;
            if (c->build_host[4] & FLAG_NONFINITE) return refuse_broken_input(c, s);
            memcpy(c->species_host, c->build_host + 8, sizeof c->species_host);
            int64_t total;
            memcpy(&total, c->build_host + 2, sizeof total);
            done = c->build_host[1] == 0 && total <= c->nbr_cap;
            if (done) { c->n_entries = total; c->n_long = c->build_host[LONG_WORD]; }
        }
        if (done) {
            mark_end(c, MARK_BUILD, s);
            return MLIP_OK;
        }
    }
    if (rel) {
        k_neighbors_rel<false, int32_t><<<blocks_for(n * 32, 256), 256, 0, s>>>(n, g, rl * rl, c->pos4, relpos, c->cell_start, c->nbr_count, nullptr, nullptr, 0, c->status, near2, c->nbr_near, c->user_of, (int32_t)c->n_owned);
    } else
        k_neighbors<false><<<blocks_for(n * 32, 256), 256, 0, s>>>(n, g, rl * rl, c->pos4, c->cell_start, c->nbr_count, nullptr, nullptr, 0, c->status, near2, c->nbr_near, c->user_of, (int32_t)c->n_owned);
    c->launches += 1 + exclusive_scan<int32_t, int64_t>(c->nbr_count, c->nbr_off, n, c->scan_tmp, s);
    MLIP_CUDA_TRY(c, cudaGetLastError());
    if (allow_sync_grow) {
        MLIP_CUDA_TRY(c, cudaMemsetAsync(c->build_word + LONG_WORD, 0, sizeof(int), s));
        k_count_long<<<blocks_for(n, 256), 256, 0, s>>>(n, c->nbr_near, c->build_word + LONG_WORD);
        c->launches += 1;
        MLIP_CUDA_TRY(c, cudaMemcpyAsync(c->total_host, c->nbr_off + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        MLIP_CUDA_TRY(c, cudaMemcpyAsync(c->build_host, c->build_word, sizeof(int) * mlip_ctx::BUILD_WORDS, cudaMemcpyDeviceToHost, s));
        MLIP_CUDA_TRY(c, cudaStreamSynchronize(s));
        if (c->build_host[4] & FLAG_NONFINITE) return refuse_broken_input(c, s);
        memcpy(c->species_host, c->build_host + 8, sizeof c->species_host);
        c->n_entries = *c->total_host;
        c->n_long = c->build_host[LONG_WORD];
        if (c->n_entries > c->nbr_cap) {
            int64_t want = c->n_entries + c->n_entries / 8 + 1024;
            if (c->nbr) { cudaFree(c->nbr); c->resident -= entry_bytes * c->nbr_cap; c->nbr = nullptr; c->nbr_cap = 0; }
            MLIP_CUDA_TRY(c, cudaMalloc(&c->nbr, entry_bytes * want));
            c->nbr_cap = want;
            c->resident += entry_bytes * want;
            nbr16 = reinterpret_cast<uint16_t *>(c->nbr);
        }
    }
    if (rel && list16)
        k_neighbors_rel<true, uint16_t><<<blocks_for(n * 32, 256), 256, 0, s>>>(n, g, rl * rl, c->pos4, relpos, c->cell_start, c->nbr_count, c->nbr_off, nbr16, c->nbr_cap, c->status, near2, c->nbr_near, c->user_of, (int32_t)c->n_owned);
    else if (rel)
        k_neighbors_rel<true, int32_t><<<blocks_for(n * 32, 256), 256, 0, s>>>(n, g, rl * rl, c->pos4, relpos, c->cell_start, c->nbr_count, c->nbr_off, c->nbr, c->nbr_cap, c->status, near2, c->nbr_near, c->user_of, (int32_t)c->n_owned);
    else
        k_neighbors<true><<<blocks_for(n * 32, 256), 256, 0, s>>>(n, g, rl * rl, c->pos4, c->cell_start, c->nbr_count, c->nbr_off, c->nbr, c->nbr_cap, c->status, near2, c->nbr_near, c->user_of, (int32_t)c->n_owned);
    c->launches += 1;
    mark_end(c, MARK_BUILD, s);
    MLIP_CUDA_TRY(c, cudaGetLastError());
    return MLIP_OK;
}

// The lists cannot be exported while the status word says that the last in-step rebuild did not complete them.  Leaves the number of
// entries in total_host.
static int lists_whole(mlip_ctx *c, cudaStream_t s) {
    MLIP_CUDA_TRY(c, cudaMemcpyAsync(c->status_host, c->status, sizeof(int), cudaMemcpyDeviceToHost, s));
    MLIP_CUDA_TRY(c, cudaMemcpyAsync(c->total_host, c->nbr_off + c->n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    MLIP_CUDA_TRY(c, cudaStreamSynchronize(s));
    if (*c->status_host & FLAG_NONFINITE) { c->err = "neighbor export: the configuration is broken (see mlip_sync_status)"; return MLIP_ERR_NONFINITE; }
    if (*c->status_host & FLAG_NEIGHBOR_OVERFLOW) { c->err = "neighbor export: the last rebuild overflowed the list (see mlip_sync_status)"; return MLIP_ERR_NEIGHBOR_OVERFLOW; }
    return MLIP_OK;
}

// Keys, scan of the list lengths, lists; if the caller's array cannot hold them, the segments only.  `counts` [n * C] and `tmp` (scan_tmp_items(n * C)) are scratch;
// the keys go to cell_of, which is read during list builds only.
static int export_lists(mlip_ctx *c, int64_t *seg_ptr, int32_t *nbr, int64_t capacity, int64_t *n_entries_host, int32_t *counts, int64_t *tmp, cudaStream_t s) {
    const int64_t n = c->n;
    const int C = c->cfg.n_species;
    if (n_entries_host) *n_entries_host = *c->total_host;
    const bool room = nbr && *c->total_host <= capacity;
    k_export_keys<<<blocks_for(n, 256), 256, 0, s>>>(n, c->pos4, c->user_of, c->nbr_off, c->cell_of, counts);
    c->launches += 2;
    if (room) {
        c->launches += exclusive_scan<int32_t, int64_t>(counts, seg_ptr, n, tmp, s, C);
        k_export_fill<<<blocks_for(n * 32, 256), 256, 0, s>>>(n, C, c->nbr_off, list_view(c), c->cell_of, seg_ptr, nbr);
    } else {
        k_export_count<<<blocks_for(n * 32, 256), 256, 0, s>>>(n, C, c->nbr_off, list_view(c), c->cell_of, counts);
        c->launches += exclusive_scan<int32_t, int64_t>(counts, seg_ptr, n * C, tmp, s);
    }
    MLIP_CUDA_TRY(c, cudaGetLastError());
    MLIP_CUDA_TRY(c, cudaStreamSynchronize(s));
    if (!room) {
        c->err = "neighbor export: capacity too small";
        return MLIP_ERR_NEIGHBOR_OVERFLOW;
    }
    return MLIP_OK;
}

int launch_export(mlip_ctx *c, int64_t *seg_ptr, int32_t *nbr, int64_t capacity, int64_t *n_entries_host, cudaStream_t s) {
    const int whole = lists_whole(c, s);
    if (whole != MLIP_OK) return whole;
    // The source set of the list builds is dead between builds and holds the scratch (device allocations here stalled the call
    // by up to 10 ms): n * C <= 8 n counts in the 32 n bytes of pos4_src, n * C / 4,096 + 3 sums in the 24 n bytes of vel_src.
    static_assert(sizeof(double4) >= MAX_SPECIES * sizeof(int32_t) && SCAN_TILE >= 8 * MAX_SPECIES, "export scratch");
    return export_lists(c, seg_ptr, nbr, capacity, n_entries_host, reinterpret_cast<int32_t *>(c->pos4_src), reinterpret_cast<int64_t *>(c->vel_src), s);
}

}  // namespace mlip

// ---- allocation-free variant of the canonical export ----
//
// For callers that must not allocate device memory while they run: code inside a region where
// cudaMalloc would serialise or fail (a latency-critical MD loop that owns a fixed memory budget, a
// plug-in running under a host application whose allocator it may not touch), or a process whose
// device memory is already fully committed.  The two temporaries of the export (per-(atom, species)
// counts and the partial sums of the prefix scan) live in a file-scope device array instead of
// fresh cudaMalloc blocks.  Every GPU that loads the library holds the array until the process exits.
namespace mlip {

constexpr int64_t NOALLOC_MAX_SEGMENTS = 1 << 20;   // n_atoms * n_species accepted by the entry point
constexpr size_t NOALLOC_COUNT_BYTES = ((sizeof(int32_t) * (NOALLOC_MAX_SEGMENTS + 1) + 255) / 256) * 256;
constexpr size_t NOALLOC_SCAN_ITEMS = NOALLOC_MAX_SEGMENTS / SCAN_TILE + 3;
constexpr size_t NOALLOC_BYTES = NOALLOC_COUNT_BYTES + sizeof(int64_t) * NOALLOC_SCAN_ITEMS;   // about 4 MiB

static __device__ __align__(256) unsigned char g_export_scratch[NOALLOC_BYTES];

// In host code `g_export_scratch` is only a handle for the runtime, not a device address; the
// address a kernel may use comes from cudaGetSymbolAddress, asked once per device with that device
// current.  Slot d caches device d's answer.  The cache is plain host state: fill it from one host thread at a time,
// and a cudaDeviceReset() of that device invalidates the cached address (the library is not meant to outlive one).
static void *g_export_scratch_addr[64] = {nullptr};

static int export_scratch_for_current_device(mlip_ctx *c, void **out) {
    int dev = -1;
    MLIP_CUDA_TRY(c, cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) { c->err = "device ordinal out of range for the static scratch table"; return MLIP_ERR_UNSUPPORTED; }
    if (!g_export_scratch_addr[dev]) {
        void *p = nullptr;
        MLIP_CUDA_TRY(c, cudaGetSymbolAddress(&p, g_export_scratch));
        g_export_scratch_addr[dev] = p;
    }
    *out = g_export_scratch_addr[dev];
    return MLIP_OK;
}

// The same export as launch_export, with the temporaries taken from the static
// array.  Every scratch word that is read (counts of all n * C segments, the scan's tile sums) is
// written earlier in the same call, so nothing has to be cleared between calls; two calls whose
// kernels overlap on the GPU (different streams or contexts on one device) would race on it.
int launch_export_noalloc(mlip_ctx *c, int64_t *seg_ptr, int32_t *nbr, int64_t capacity, int64_t *n_entries_host, cudaStream_t s) {
    if (c->n * c->cfg.n_species > NOALLOC_MAX_SEGMENTS) {
        c->err = "mlip_get_neighbors_noalloc: n_atoms * n_species exceeds 1048576 (the static scratch size); use mlip_get_neighbors";
        return MLIP_ERR_UNSUPPORTED;
    }
    void *base = nullptr;
    int rc = lists_whole(c, s);
    if (rc != MLIP_OK) return rc;
    if ((rc = export_scratch_for_current_device(c, &base)) != MLIP_OK) return rc;
    return export_lists(c, seg_ptr, nbr, capacity, n_entries_host, reinterpret_cast<int32_t *>(base),
                        reinterpret_cast<int64_t *>(static_cast<unsigned char *>(base) + NOALLOC_COUNT_BYTES), s);
}

}  // namespace mlip
