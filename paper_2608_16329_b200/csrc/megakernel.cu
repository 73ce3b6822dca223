// The fused evaluation kernel (megakernel.cuh): weights, launch.
#include <algorithm>
#include <new>
#include <vector>

#include "list_form.cuh"
#include "megakernel.cuh"

namespace mlip {

static_assert(LONG_LIST == NARROW_CHUNKS * 32, "lists that two atoms gather together");

// ---------------- host side ----------------
int table_smem_words(const mlip_ctx *c) { return c->cfg.n_species * (c->cfg.table_knots + 3) * K_RADIAL; }
bool tables_fit_smem(const mlip_ctx *c) {   // (the rows' 16-bit addresses, with room for a reserved kilobyte in front, are the tighter limit)
    return Layout<2>::FIXED + table_smem_words(c) <= SMEM_LIMIT_WORDS && 4 * table_smem_words(c) + 2048 <= 65536;
}

static float pow2f(int e) { return ldexpf(1.f, e); }

// The tensor-memory image of the weights, one thread per word: A fragments; k-step ks, lane (g, t), register r holds row
// 16 m + g + 8 (r & 1) and the k pair (n, n + 8) with n = 16 ks + t + 4 (r >> 1)  (see act_store).
struct HeadScales { float w[MAX_SPECIES][HEAD_L]; };
__global__ void k_pack_head(const double *__restrict__ nets, HeadScales sc, uint32_t *__restrict__ image) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x, s = blockIdx.y;
    const int lane = (idx >> 2) & 31, col = 4 * ((idx >> 7) % (TM_VT / 4)) + (idx & 3), quarter = (idx >> 7) / (TM_VT / 4);
    const int g = lane >> 2, t = lane & 3, r = col & 3, row = g + 8 * (r & 1), n = t + 4 * (r >> 1);
    int L, m = quarter, ks;
    bool reverse = col >= TM_BWD;
    if (col < TM_FWD) { L = 0; ks = col >> 3; }
    else if (col < TM_BWD) { L = 1 + (col - TM_FWD) / 32; ks = ((col - TM_FWD) & 31) >> 3; }
    else if (col < TM_BWD0) { L = 1 + (col - TM_BWD) / 32; ks = ((col - TM_BWD) & 31) >> 3; }
    else { L = 0; m += 4 * ((col - TM_BWD0) / 32); ks = ((col - TM_BWD0) & 31) >> 3; }
    const int in = L == 0 ? N_INV : HEAD_H;
    const double *W = nets + (size_t)s * HEAD_NET + (L == 0 ? 0 : N_INV * HEAD_H + HEAD_H + (L - 1) * (HEAD_H * HEAD_H + HEAD_H));
    // forward: A[m][k] = W[m][k]; reverse: A[m][k] = W[k][m]
    const double *src = reverse ? W + (size_t)(16 * ks + n) * in + 16 * m + row : W + (size_t)(16 * m + row) * in + 16 * ks + n;
    uint32_t hi, lo;
    split_h2((float)src[0] * sc.w[s][L], (float)src[reverse ? 8 * in : 8] * sc.w[s][L], hi, lo);
    image[(size_t)s * HP_TOTAL + idx] = col & 4 ? lo : hi;
}

// (after build_tables: the first layer is scaled to match the tables)
int upload_head(mlip_ctx *c, const double *w) {
    const int C = c->cfg.n_species;
    std::vector<double> scaled;    // the networks with the first layer's columns equalised
    std::vector<float> consts;     // [C][HC_USED]
    try { scaled.assign(w, w + (size_t)C * HEAD_NET); consts.resize((size_t)C * HC_USED); } catch (const std::bad_alloc &) { return MLIP_ERR_OOM; }
    HeadScales scales;
    for (int s = 0; s < C; ++s) {
        const double *layer[HEAD_L], *out = scaled.data() + (size_t)s * HEAD_NET;
        int in_of[HEAD_L];
        for (int L = 0, in = N_INV; L < HEAD_L; ++L, in = HEAD_H) { layer[L] = out; in_of[L] = in; out += in * HEAD_H + HEAD_H; }
        float *hc = consts.data() + (size_t)s * HC_USED;
        // The tables carry 2^table_exp per channel, the moments too, the invariants once (l = 0) or squared: the weights take the
        // inverse.  Then every column is brought to a largest weight in [1/2, 1) and its invariant multiplied by what was
        // divided out, so that the values in one contraction are compared by what they contribute.
        double *first = scaled.data() + (size_t)s * HEAD_NET, most_of[N_INV] = {0.0};
        for (int o = 0; o < HEAD_H; ++o)
            for (int q = 0; q < N_INV; ++q) most_of[q] = std::max(most_of[q], fabs(first[(size_t)o * N_INV + q]));
        for (int q = 0; q < N_INV; ++q) {
            int e = 0;
            if (most_of[q] > 0.0) frexp(most_of[q], &e);
            const int te = c->table_exp[s * K_RADIAL + q % K_RADIAL] * (q < K_RADIAL ? 1 : 2);
            const int ce = std::max(-126, std::min(126, e - te));
            hc[HC_CS + q] = pow2f(ce);
            most_of[q] = ldexp(1.0, -te - ce);
        }
        for (int o = 0; o < HEAD_H; ++o)
            for (int q = 0; q < N_INV; ++q) first[(size_t)o * N_INV + q] *= most_of[q];
        // powers of two: the weights of a layer to below 2^14
        float *wscale = scales.w[s];
        for (int L = 0; L < HEAD_L; ++L) {
            double most = 0.0;
            for (int q = 0; q < HEAD_H * in_of[L]; ++q) most = std::max(most, fabs(layer[L][q]));
            int e = 0;
            if (most > 0.0) frexp(most, &e);
            wscale[L] = pow2f(std::min(14 - e, 60));
            hc[HC_WS + L] = 1.f / wscale[L];
        }
        for (int L = 0; L < HEAD_L; ++L)
            for (int o = 0; o < HEAD_H; ++o) hc[L * HEAD_H + o] = (float)layer[L][(size_t)in_of[L] * HEAD_H + o];
        for (int o = 0; o < HEAD_H; ++o) hc[HC_WOUT + o] = (float)out[o];
        hc[HC_BOUT] = (float)out[HEAD_H];
    }
    const size_t bytes = sizeof(uint32_t) * (size_t)C * HP_TOTAL, net_bytes = sizeof(double) * (size_t)C * HEAD_NET;
    double *nets = nullptr;
    MLIP_CUDA_TRY(c, cudaMalloc(&c->head_w, bytes));
    MLIP_CUDA_TRY(c, cudaMalloc(&nets, net_bytes));
    cudaError_t e = cudaMemcpy(nets, scaled.data(), net_bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_pack_head<<<dim3(4 * TM_VT * 32 / 256, C), 256>>>(nets, scales, c->head_w);
        c->launches += 1;
        e = cudaMemcpy2D(c->head_w + HP_TMEM, sizeof(uint32_t) * HP_TOTAL, consts.data(), sizeof(float) * HC_USED, sizeof(float) * HC_USED, C, cudaMemcpyHostToDevice);
    }
    cudaFree(nets);
    if (e != cudaSuccess) { c->err = cudaGetErrorString(e); return MLIP_ERR_CUDA; }
    c->resident += bytes;
    return MLIP_OK;
}

// Deterministic mode: integer sums -> the float / double outputs the rest of the library reads; the sums start the next evaluation at zero.
__global__ void k_fixed_finish(int64_t n, long long *force_fx, const long long *acc_fx, float4 *force, double *acc, unsigned long long *stamp) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    allow_next();
    wait_previous();
    if (i < n) {
        const double inv = 1.0 / (double)FORCE_FX;
        force[i] = make_float4((float)((double)force_fx[3 * i] * inv), (float)((double)force_fx[3 * i + 1] * inv),
                               (float)((double)force_fx[3 * i + 2] * inv), 0.f);
        force_fx[3 * i] = force_fx[3 * i + 1] = force_fx[3 * i + 2] = 0;
    }
    if (i == 0) {
        acc[ACC_ENERGY] = (double)acc_fx[0] / ENERGY_FX;
        for (int q = 0; q < 9; ++q) acc[ACC_VIRIAL + q] = (double)acc_fx[1 + q] / VIRIAL_FX;
    }
    stamp_end(stamp);
}

// Whether two atoms of a warp go through the pair loops one after the other.  Side by side they are the faster ones where their lists fit the queue
// together, up to LONG_LIST entries each; with longer ones they are gathered one by one as well, no batch is saved, and from some 110 pairs on
// warps of both kinds, which then share an SM, hold each other up.  One evaluation of some 100,000 atoms in us, side by side / one after the
// other: random positions of 54 pairs an atom 667 / 671, 63 734 / 735, 72 823 / 801, 81 886 / 858, 109 1564 / 1057, 118 2632 / 1203, 163 2131 / 1529; crystals
// of 42 pairs 494 / 512, 54 574 / 585, 78 846 / 853, 86 995 / 964, 113 1215 / 1153, 131 1506 / 1367, 158 1534 / 1377, 221 2317 / 2123.
// Asked of the last synchronising build's lists.  Reproducible runs must not depend on when that was: they ask the density of the box.
static bool long_lists(const mlip_ctx *c) {
    if (c->cfg.force_mode != 1) return lists_are_long(c->n_long, c->n_owned);
    const double r = c->cfg.r_cut + 0.5 * c->cfg.skin, volume = c->grid.box[0] * c->grid.box[1] * c->grid.box[2];
    return lists_expected_long((double)c->n / volume * (4.0 / 3.0 * 3.14159265358979 * r * r * r));
}

int launch_megakernel(mlip_ctx *c, cudaStream_t s) {
    const int64_t n = c->n;
    const bool det = c->cfg.force_mode == 1;
    const EvalBlocks blk = next_eval_blocks(c);
    if ((!c->force_cleared || c->captured) && !det) {   // (k_fixed_finish keeps the integer sums clear)
        c->mark_open = false;
        MLIP_CUDA_TRY(c, cudaMemsetAsync(c->force, 0, sizeof(float4) * n, s));
    }
    if (c->captured) MLIP_CUDA_TRY(c, cudaMemsetAsync(blk.use, 0, LAUNCH_CLEAR_BYTES, s));
    const bool in_smem = tables_fit_smem(c);
    const int tab_words = in_smem ? table_smem_words(c) : 0;
    const int shape = in_smem && n < ONE_PER_WARP_BELOW_ATOMS ? 0 : long_lists(c) ? 2 : 1;   // one atom per warp, two side by side, two one after the other
    const int apw = shape == 0 ? 1 : 2;
    const size_t smem_bytes = sizeof(float) * (size_t)((apw == 1 ? Layout<1>::FIXED : Layout<2>::FIXED) + tab_words);
    const int C = c->cfg.n_species, tile_atoms = GW * apw;
    int64_t tiles[MAX_SPECIES], all = 0;
    for (int q = 0; q < C; ++q) all += tiles[q] = (c->species_host[q + 1] - c->species_host[q] + tile_atoms - 1) / tile_atoms;
    const int blocks = (int)std::min<int64_t>(all, (int64_t)c->n_sm);
    const MegaKernel kernel = shape == 0 ? mega_one(det, c->list16) : shape == 2 ? mega_apart(in_smem, det, c->list16) : !in_smem ? mega_two_global(det, c->list16)
                            : det ? mega_two_fixed(c->list16) : mega_two(c->list16);
    const int ready = 1 << (2 * shape + (c->list16 ? 1 : 0));
    if (!(c->kernel_ready & ready)) {
        // A limit of the kernel, shared by every context of the process: the same whatever this one's tables need.
        const cudaError_t e = cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(float) * (in_smem ? SMEM_LIMIT_WORDS : Layout<2>::FIXED));
        if (e != cudaSuccess) { c->err = std::string("fused kernel shared memory: ") + cudaGetErrorString(e); return MLIP_ERR_CUDA; }
        c->kernel_ready |= ready;
    }
    KernelArgs k;
    k.n = n; k.n_species = c->cfg.n_species; k.grid = c->grid; k.rc2 = c->cfg.r_cut * c->cfg.r_cut; k.tab = c->tab;
    k.pos4 = c->pos4; k.center_order = c->center_order;
    k.nbr_off = c->nbr_off; k.nbr_near = c->nbr_near; k.far_flag = c->far_flag; k.nbr = c->nbr; k.nbr16 = reinterpret_cast<const uint16_t *>(c->nbr); k.cell_id = c->cell_id; k.cell_start = c->cell_start;
    k.nbr_cap = c->nbr_cap; k.head_pack = c->head_w; k.force = c->force; k.e_atom = c->e_atom;
    k.force_fx = c->force_fx; k.acc_fx = reinterpret_cast<long long *>(blk.use + LB_ACC_FX);
    k.acc = blk.use + LB_ACC; k.pair_counter = reinterpret_cast<unsigned long long *>(blk.use + LB_PAIR);
    k.status = c->status; k.tile_counter = reinterpret_cast<int *>(blk.use);
    k.clear_block = blk.clear; k.species_dev = c->captured ? c->species_start : nullptr;
    // CTAs in proportion to the species' tiles, at least one to a species that has any.  (One evaluation in us with the CTAs dealt out to the
    // species in turn / in proportion: 864 atoms 90:5:5 46 / 23.5, 6,912 atoms 80 / 66, 13,824 atoms 47:12:41 116 / 96; six equal
    // species, where in turn left some with more tiles than groups, 864 atoms 35.7 / 28.4, 23,328 atoms 221 / 198.)
    // From 64 tiles a CTA on, rare species (below half the mean) round up: their CTAs end early and join a species that many work on,
    // where rounded down they end late and all the others stage the rare species for a last tile (90:5:5, all CTAs in
    // order / rounded down / up, us: 202,612 atoms 1326 / 1344 / 1305, 415,292 2676 / 2689 / 2651, 1,000,188 6394 / 6364 / 6330).
    int64_t weight[MAX_SPECIES], total = 0, before = 0;
    for (int q = 0; q < C; ++q) total += weight[q] = tiles[q] > 0 ? std::max<int64_t>(tiles[q], 2 * all / blocks) : 0;
    int up[MAX_SPECIES] = {0}, shared = blocks, fixed = 0;   // CTAs of rare species, of the others
    const int64_t whole = total;
    for (int q = 0; q < C; ++q) {
        if (all < (int64_t)64 * blocks || tiles[q] == 0 || 2 * C * tiles[q] >= all) continue;
        up[q] = (int)((weight[q] * blocks + whole - 1) / whole);   // (together at most blocks / 2 + C of them)
        shared -= up[q]; total -= weight[q];
    }
    for (int q = 0; q <= MAX_SPECIES; ++q) {
        k.species_start[q] = c->species_host[std::min(q, C)];
        k.first_cta[q] = q < C ? fixed + (int)(before * shared / total) : blocks;
        if (q < C) up[q] > 0 ? (void)(fixed += up[q]) : (void)(before += weight[q]);
    }
    k.stamp = timed_begin(c, MARK_KERNEL, s);
    k.early = !c->lists_fresh;   // (the kernel reads the lists before it waits)
    MLIP_CUDA_TRY(c, launch_after_if(k.early, kernel, blocks, NW * 32, smem_bytes, s, k, tab_words));
    c->lists_fresh = c->force_cleared = false;
    set_eval_block(c, blk.use);
    if (det) {
        MLIP_CUDA_TRY(c, launch_after(k_fixed_finish, (unsigned)((n + 255) / 256), 256, 0, s, n, c->force_fx, c->acc_fx, c->force, c->acc, k.stamp));
        c->launches += 1;
    }
    timed_end(c, MARK_KERNEL, s);
    c->launches += 1;
    return MLIP_OK;
}

}  // namespace mlip
