// The fused evaluation kernel (Section 3.4.1 "mega-fusion": Eq. 1-10 in one launch; every
// per-pair and per-atom intermediate lives in registers or shared memory, and the radial and
// angular features are recomputed in the derivation stage instead of being kept).
//
// Work decomposition
//   One persistent CTA of 16 warps per SM, organised as two independent groups of 8 warps.  The CTA
//   walks through the central species in order; for each it stages that species' radial tables
//   (one per neighbor species) and head constants in shared memory, then each group takes tiles of
//   16 (small systems: 8) central atoms of that species from a global counter (each warp encodes and
//   derives two of them, side by side in its pair loops where lists are short) and runs them on its own,
//   synchronising only inside the group (named barriers), so that one group's latency-bound head
//   overlaps the other group's pair loops.
//   Encoding    The warp scans the atom's list (lane = entry), queues the pairs inside r_cut in
//               shared memory, and every 32 queued pairs evaluates harmonics (Eq. 3) and the
//               spline basis with lane = pair.  The moment P_i = H^T G (Eq. 4, 16 x n times
//               n x 32) is accumulated on the tensor pipe: mma.sync m16n8k16 with both operands as fp16
//               hi + lo pairs (three products, ~2^-22 relative, fp32 accumulate), the
//               radial values g being evaluated straight into the B fragments.  P_i waits
//               in tensor memory for the derivation.
//   Invariants  Eq. 5 from the accumulator fragments by three xor-shuffles.
//   Regression  Eq. 6 forward and reverse for the atoms of the tile at once as W X^T on the tensor pipe
//               (mma.sync m16n8k16, fp16 operands in hi + lo pairs: 22 significant bits, fp32 accumulate); a
//               warp keeps its 16 neurons x 8 atoms in accumulator fragments from layer to layer and passes
//               the activations on through shared memory in B-fragment order, one barrier per layer.
//               The current species' weights live in tensor memory (tcgen05.alloc / st / ld), split already: a
//               warp fetches 32 registers of A fragments in one instruction, off the L1/shared-memory pipe.
//   Derivation  W_i (Eq. 7) is the accumulator fragment of P_i scaled in place: by construction
//               of the channel permutation it already is the B fragment of the next contraction.
//               [V; T] = [G; G'] W^T (Eq. 9 and the re-associated Eq. 8 term, U_i never formed)
//               on the tensor pipe, 16 pairs per tile; results are transposed through tensor
//               memory to lane = pair for the projection of Eq. 10 and the scatter.
// Everything that is not a contraction (geometry, harmonics, splines, projection) stays on the
// fp32 pipe; positions are differenced in fp64.
// Lists come in two parts (neighbor.cu): entries that were within r_cut + skin / 2 at build time first, the rest
// behind them; the far part cannot reach r_cut before some atom has moved skin / 4, and is skipped until the
// integrator raises far_flag.
// Three-term products: both operands of every contraction are split into fp16 hi + lo (22 significant bits, the same as two
// TF32 terms) and A_lo B_hi + A_hi B_lo + A_hi B_hi is accumulated in fp32.  fp16 halves the tensor instructions and the fragment
// registers of TF32.  Its narrow exponent range (full precision over 2^18 below the largest scaled value, an absolute error of 2^-40
// of it further down) is met by exact powers of two: the radial tables are stored scaled per central species and channel
// (tables.cu) with the regression's first layer scaled to match and equalised per input (upload_head), and the activations (per atom
// and 16 neurons) and W_i (per atom) carry scales taken from their largest value, which fp32 takes back.
#pragma once
#include <cuda_fp16.h>

#include "common.cuh"
#include "pair_math.cuh"

namespace mlip {

constexpr int GW = 8;         // warps per group; a tile is GW x APW atoms, APW = atoms per warp (1 or 2)
constexpr int NG = 2;         // groups per CTA
constexpr int NW = NG * GW;   // warps per CTA
constexpr int J_BITS = 28;    // queue entries pack the neighbor index (low 28 bits) with its species
constexpr int ST_STRIDE = 20; // encoding hand-over: h as 8 words hi + 8 words lo (fp16 pairs), 4 b (80 bytes: conflict-free for ldmatrix and STS.128)
constexpr int BS_STRIDE = 12; // derivation hand-over: 4 b, 4 b', row addresses
constexpr int X_STRIDE = 132; // dE/dG per atom

// Radial table rows (32 channels, 128 bytes, read by both pair loops) are stored with their eight 16-byte chunks permuted: chunk
// c of row r sits at position c ^ table_swizzle(r).  Lanes that read the same chunk of rows with different r mod 4 then hit
// different bank groups; every pair uses four consecutive rows, one of each residue, and the pair loops take them in an
// order that gives the lanes of a load different residues (RowOffsets).  Without that the rows of a load are random and
// collide: 6 instead of 4 wavefronts per pair in the derivation, and a shuffle per value in the encoding.
static_assert(K_RADIAL == 32, "a table row is eight 16-byte chunks");
constexpr int SCR_WORDS = 32 * ST_STRIDE + 32 * 4;              // scratch of a warp: hand-over rows, table row addresses
static_assert(32 * BS_STRIDE <= SCR_WORDS && N_INV <= X_STRIDE, "the derivation's hand-over must fit the encoding's, the invariants the row of dE/dG");
// Regression buffers of a group.  Activations are kept as B fragments: per 16-input k-step, atom row and quad lane one
// 16-byte vector {b0 hi, b0 lo, b1 hi, b1 lo} of fp16 pairs (see act_store).
constexpr int ACT_KSTEP = 32 * 4;                               // words per k-step
constexpr int XS_WORDS = (N_INV / 16) * ACT_KSTEP;              // split invariants of eight atoms (written before the group's barrier: space of their own)
constexpr int ZS_WORDS = (HEAD_H / 16) * ACT_KSTEP;             // one layer's activations of eight atoms
constexpr int PF_IDX = 160;                                     // neighbor indices prefetched per coming atom
constexpr int PF_CS = 96;                                       // compact lists: the codes take 81 words at most, the 27 cell bases sit here
static_assert(PF_IDX / 2 + 1 <= PF_CS && PF_CS + 27 <= PF_IDX, "prefetch buffer layout for compact lists");
constexpr int PF_WORDS = PF_IDX + 4;                            // + {atom, list start (2 words), list length}
static_assert(2 * 2 * ZS_WORDS <= GW * SCR_WORDS, "layer activations alias the scratch of the group's warps");
// Head constants of the current species: biases, w_out, b_out, then the powers of two of the fp16 scaling:
//   a product with layer L's weights is unscaled by HC_WS[L], besides the scale of the activations
//   the invariants enter, and dE/dG leaves, times HC_CS[input]: the powers of two that equalise the first layer's columns
constexpr int HC_WOUT = HEAD_L * HEAD_H, HC_BOUT = HC_WOUT + HEAD_H, HC_WS = HC_BOUT + 1, HC_CS = HC_WS + HEAD_L, HC_USED = HC_CS + N_INV;
constexpr int HC_WORDS = (HC_USED + 15) / 16 * 16;
constexpr int CTL_WORDS = 16;   // per group {tile, tile after it}; tensor-memory base; the species' starts
static_assert(5 + MAX_SPECIES + 1 <= CTL_WORDS, "control words");
// Systems below this size take tiles of 8 atoms, one per warp: with few tiles per SM the chain through one tile is what counts
// (one evaluation in us with 8- / 16-atom tiles, 6 species: 256 atoms 26 / 35, 864 29 / 36, 4,000 55 / 53, 6,912 85 / 90, 10,976 115 / 125,
// 16,384 166 / 162, 32,000 292 / 271, 131,072 1125 / 1063; one species: 686 atoms 26 / 28, 4,394 45 / 43, 8,192 78 / 73, 11,664 95 / 103,
// 16,000 128 / 133, 31,250 241 / 224, 65,536 472 / 433; three: 10,976 97 / 106, 16,384 140 / 137.  In between it depends on how full the
// last round of tiles is).  Tables in global memory (seven species or more, or many knots): compiled with 16-atom tiles only; 8-atom ones
// would be faster below the same size (8 species: 864 atoms 27 / 40, 10,976 122 / 140, 16,384 183 / 181, 131,072 1215 / 1212).
constexpr int64_t ONE_PER_WARP_BELOW_ATOMS = 12000;
// Shared memory per tile shape.  Two atoms per warp halve the regression's barriers, weight fetches and idle time per atom
// (each warp owns 16 neurons x 8 atoms of a 16-atom tile instead of half of the warps owning an 8-atom tile); one atom per warp
// spreads a small system over more SMs.
template <int APW>
struct Layout {
    static constexpr int NA = GW * APW;                         // atoms per tile
    static constexpr int POOL = APW == 1 ? 160 : 256;           // pair queue of a warp, shared by its atoms, kept from encoding to derivation
    static constexpr int Q_WORDS = 4 * POOL;
    static constexpr int SX = NA * X_STRIDE;                    // dE/dG
    static constexpr int US = NA / 2 * (HEAD_H / 16);           // one layer's activation scales (see act_store_scaled)
    static constexpr int SC = 2 * US + NA;                      // two layers of them, then the invariants' (see split_invariants)
    static constexpr int EP = 4 * NA;                           // E_i partial sums of the four m-tiles
    static constexpr int GROUP = APW * XS_WORDS + SX + SC + EP;
    static constexpr int INFO = 4 * APW;                        // per warp: {atom, queued pairs, queue start, -} of its atoms, from encoding to derivation
    static constexpr int WARP = Q_WORDS + SCR_WORDS + APW * PF_WORDS + INFO;
    static constexpr int FIXED = NG * GROUP + NW * WARP + HC_WORDS + CTL_WORDS;
};
constexpr int SMEM_LIMIT_WORDS = 227 * 1024 / 4 - 256;

// Pre-packed head weights per species (32-bit words): the tensor-memory image, [quarter][column / 4][lane][4], followed by
// the HC_USED constants (as fp32).  Quarter q holds m-tile q (16 neurons) of every forward layer and of the hidden layers'
// reverse pass, and m-tiles q, q + 4 (16 inputs each) of the first layer's reverse pass.  A 16-wide k-step of one m-tile
// takes eight columns: the A fragment's four registers of fp16 pairs, hi then lo.
//   columns [  0,  64)  forward, first layer: 8 k-steps
//           [ 64, 160)  forward, hidden layers: 3 x 4 k-steps
//           [160, 256)  reverse, hidden layers: 3 x 4 k-steps
//           [256, 320)  reverse, first layer: 2 m-tiles x 4 k-steps
//           [320, 448)  V and T on their way from fragments to lane = pair: 32 columns per warp of the quarter; before that
//                       the moment P of the warp's second atom waits there for its derivation
//           [448, 512)  P of the warp's first atom: 16 columns per warp of the quarter
constexpr int TM_FWD0 = 0, TM_FWD = 64, TM_BWD = 160, TM_BWD0 = 256, TM_VT = 320, TM_P = 448;
constexpr int HP_TMEM = 4 * TM_VT * 32;
constexpr int HP_TOTAL = HP_TMEM + (HC_USED + 3) / 4 * 4;

// The PTX ISA's approximations in their .ftz forms, which take subnormal arguments and results for zero.  Such arguments do not occur here
// (squared distances of atoms that do not coincide, 1 + exp(-x)) or change nothing (an exponential below 2^-126 adds nothing to 1).
// One evaluation with rsqrtf, __expf and __fdividef / with these: 1,000,188 atoms 7479 / 7439 us, 256,000 with 54 pairs 1634 / 1621.
__device__ __forceinline__ float fast_rsqrt(float x) { float y; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float fast_rcp(float x) { float y; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float fast_exp2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
// SiLU and its derivative.  exp(-x) as 2^(-x log2 e) through the fast exponential: its error scales with |x| 2^-24 and
// enters the sigmoid damped by s (1 - s), far below fp32 rounding of the surrounding sums.
__device__ __forceinline__ float silu_f(float x, float &dsilu) {
    const float s = fast_rcp(1.0f + fast_exp2(x * -1.44269504f));
    dsilu = s * (1.0f + x * (1.0f - s));
    return x * s;
}

// Two fp32 FMAs in one instruction (sm_100 packed arithmetic): d = a * b + c per component.  Halves the issue slots
// of the spline evaluations, whose operands already sit in register pairs from 128-bit loads.
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    unsigned long long ra, rb, rc, rd;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rc) : "f"(c.x), "f"(c.y));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(rd) : "l"(ra), "l"(rb), "l"(rc));
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(rd));
    return d;
}

__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    unsigned long long ra, rb, rd;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(ra), "l"(rb));
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(rd));
    return d;
}
// x, y -> fp16 pairs hi, lo with hi + lo = x to 22 significant bits (x in the lower half; |x| must stay inside fp16's
// range, which the callers' power-of-two scales see to: below 2^-3 of a scaled unit lo loses bits, an absolute 2^-25).
__device__ __forceinline__ void split_h2(float x, float y, uint32_t &hi, uint32_t &lo) {
    float lx, ly;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(y), "f"(x));
    asm("{.reg .b16 h0, h1, m1; mov.b32 {h0, h1}, %2; mov.b16 m1, 0xBC00; fma.rn.f32.f16 %0, h0, m1, %3; fma.rn.f32.f16 %1, h1, m1, %4;}"
        : "=f"(lx), "=f"(ly) : "r"(hi), "f"(x), "f"(y));
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(ly), "f"(lx));
}
__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16_z(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
// The power of two 2^s with |x| 2^s < 2^15 for every |x| <= bound, and its inverse.
__device__ __forceinline__ float scale_for(float bound) {
    const int e = 268 - (int)(__float_as_uint(bound) >> 23);
    return __uint_as_float((uint32_t)(e > 253 ? 253 : e) << 23);
}
__device__ __forceinline__ float inverse_pow2(float s) { return __uint_as_float((254u << 23) - __float_as_uint(s)); }
// Two such scales at once, as bf16 halves: the inverses for the values whose upper 16 bits (sign clear) are the halves of `most`, and
// the scales from them.
__device__ __forceinline__ uint32_t inverse_scales(uint32_t most) { return (__vmaxu2(most, 0x07800780u) & 0x7f807f80u) - 0x07000700u; }
__device__ __forceinline__ uint32_t inverse_of(uint32_t w) { return 0x7f007f00u - w; }
__device__ __forceinline__ float2 unpack_bf16(uint32_t w) { return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }

// The tensor pipe truncates when it adds into its fp32 accumulator, so the energy path keeps accumulation chains short (a fresh
// accumulator per k-step, folded into the running sum by a rounded fp32 add): a long chain of same-sign terms otherwise drifts
// by ~1e-6 relative.
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Deterministic mode (force_mode = 1): every sum whose order depends on scheduling -- the force scatter across
// warps, the energy and virial totals -- is taken in integer arithmetic, which is associative, so two runs on the
// same input agree bit for bit.  Per-atom and per-pair terms are computed in a fixed order in either mode.
constexpr float FORCE_FX = 4294967296.f;        // 2^32 per eV/Angstrom
constexpr double ENERGY_FX = 4294967296.0;      // 2^32 per eV
constexpr double VIRIAL_FX = 268435456.0;       // 2^28 per eV
__device__ __forceinline__ void fixed_add3(long long *p, float x, float y, float z) {
    atomicAdd(reinterpret_cast<unsigned long long *>(p), (unsigned long long)__float2ll_rn(x * FORCE_FX));
    atomicAdd(reinterpret_cast<unsigned long long *>(p + 1), (unsigned long long)__float2ll_rn(y * FORCE_FX));
    atomicAdd(reinterpret_cast<unsigned long long *>(p + 2), (unsigned long long)__float2ll_rn(z * FORCE_FX));
}

struct KernelArgs {
    int64_t n;
    int n_species;
    CellGrid grid;
    double rc2;
    TableDesc tab;
    const double4 *pos4;
    const int32_t *center_order;
    int species_start[MAX_SPECIES + 1];   // in center_order (a step's own rebuilds do not change it)
    const int *species_dev;               // the same on the device, read instead in launches that may be replayed; else nullptr
    int first_cta[MAX_SPECIES + 1];       // the first CTA that starts on a species
    const int64_t *nbr_off;
    const int32_t *nbr_near;   // leading entries of each list that can be inside r_cut while far_flag is down
    const int *far_flag;
    const int32_t *nbr;
    const uint16_t *nbr16;     // the same array when the lists hold 16-bit cell-relative codes (L16 instantiations)
    const int32_t *cell_id;    // build-time cell of each atom (L16)
    const int32_t *cell_start; // first atom of each cell (L16)
    int64_t nbr_cap;           // entries the list array holds (range-checked builds)
    const uint32_t *head_pack;
    float4 *force;
    long long *force_fx;   // deterministic mode: forces as 2^-32 eV/Angstrom integers [N][3]
    long long *acc_fx;     // deterministic mode: energy (2^-32 eV) and virial (2^-28 eV) integers [10]
    float *e_atom;
    double *acc;
    unsigned long long *pair_counter;
    int *status;
    int *tile_counter;
    double *clear_block;       // the other evaluation block (next_eval_block)
    unsigned long long *stamp;
    bool early;                // launched to start before the kernel ahead of it has ended
};

// The radial tables of the current central species: in shared memory or, when they do not fit, in global memory (same
// layout).  Rows are numbered through the neighbor species.
struct TableView {
    const float *base;
    uint32_t saddr;   // shared-memory address of the first row (TAB_SMEM), a multiple of 128
};
template <bool TAB_SMEM>
__device__ __forceinline__ float4 table_load(const TableView &tv, uint32_t off) {   // off: row address | chunk position, see RowOffsets
    float4 v;
    if (TAB_SMEM) asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(off));
    else v = __ldg(reinterpret_cast<const float4 *>(reinterpret_cast<const char *>(tv.base) + off));
    return v;
}
static_assert(table_swizzle(2) == (table_swizzle(0) ^ 4) && table_swizzle(3) == (table_swizzle(1) ^ 4) && table_swizzle(0) == (table_swizzle(2) ^ 4), "see RowOffsets");
template <bool TAB_SMEM> constexpr int OFF_WORDS = TAB_SMEM ? 2 : 4;
// Byte addresses of a pair's four rows in the order they are taken, handed from the lane that owns the pair to the lanes that
// evaluate it: 16-bit shared-memory addresses (the tables come first in shared memory and end below 64 KB) or 32-bit offsets.
template <bool TAB_SMEM> struct RowOffsets;
template <> struct RowOffsets<true> {
    uint2 o;
    // rows first + ((turn + s) & 3), s = 0..3.  A chunk's position two steps on differs in one bit (table_swizzle(r + 2) is table_swizzle(r) ^ 4):
    // that bit travels with the addresses, so that a lane keeps the positions of two steps.
    __device__ __forceinline__ void make(const TableView &tv, int first, int turn) {
        const uint32_t order = __funnelshift_r(0x03020100u, 0x03020100u, 8 * turn);   // bytes turn, turn + 1, .. mod 4
        const uint32_t both = (tv.saddr + 128u * first) * 0x10001u;
        o.x = __byte_perm(order, 0, 0x4140) * 128u + both;
        o.y = __byte_perm(order, 0, 0x4342) * 128u + (both ^ 0x400040u);
    }
    __device__ __forceinline__ void store(float *p) const { *reinterpret_cast<uint2 *>(p) = o; }
    __device__ __forceinline__ void load(const float *p) { o = *reinterpret_cast<const uint2 *>(p); }
    // address of step s's row with the chunk position of step s & 1 (a multiple of 16 below 128) in its low bits
    __device__ __forceinline__ uint32_t at(int s, const uint32_t (&chunk)[2]) const {
        const uint32_t w = s < 2 ? o.x : o.y;
        return (s & 1 ? w >> 16 : w & 0xffffu) ^ chunk[s & 1];
    }
};
template <> struct RowOffsets<false> {
    uint4 o;
    __device__ __forceinline__ void make(const TableView &, int first, int turn) {
        o = make_uint4(128u * (first + (turn & 3)), 128u * (first + ((turn + 1) & 3)), 128u * (first + ((turn + 2) & 3)) ^ 64u, 128u * (first + ((turn + 3) & 3)) ^ 64u);
    }
    __device__ __forceinline__ void store(float *p) const { *reinterpret_cast<uint4 *>(p) = o; }
    __device__ __forceinline__ void load(const float *p) { o = *reinterpret_cast<const uint4 *>(p); }
    __device__ __forceinline__ uint32_t at(int s, const uint32_t (&chunk)[2]) const { return (s == 0 ? o.x : s == 1 ? o.y : s == 2 ? o.z : o.w) ^ chunk[s & 1]; }
};
// b[0..3] -> b[turn], b[turn + 1], .. (mod 4): spline weights in the order the rows are taken
__device__ __forceinline__ float4 rotate4(const float (&b)[4], int turn) {
    const bool r1 = turn & 1, r2 = turn & 2;
    const float c0 = r1 ? b[1] : b[0], c1 = r1 ? b[2] : b[1], c2 = r1 ? b[3] : b[2], c3 = r1 ? b[0] : b[3];
    return make_float4(r2 ? c2 : c0, r2 ? c3 : c1, r2 ? c0 : c2, r2 ? c1 : c3);
}

// Fill the warp's pair queue (room for `cap` pairs at pq) from list position `cur` on (lane = entry), up to five 32-entry chunks
// at a time with all index loads, then all position gathers, in flight together (a typical list
// of ~134 entries is one round trip).  Pairs inside r_cut are queued as {x, y, z, j | species << 28}.
// Stops when the list ends or the next group might not fit; returns the number of queued pairs
// and advances `cur`.  The first n_pref indices of the list may come from shared memory (sidx).
constexpr int WIDE_CHUNKS = 5, NARROW_CHUNKS = 3;
static_assert(WIDE_CHUNKS * 32 <= Layout<1>::POOL, "a full group must fit an empty queue");
// (a tile's second atom finds at least this much room: the first keeps at most POOL - SECOND_ROOM pairs)
constexpr int SECOND_ROOM = NARROW_CHUNKS * 32;
// Compact lists: lane q < 27 holds the first atom of the q-th cell around atom i's build-time cell; an entry's index is
// that base (one shuffle) plus the position coded in its low bits.
__device__ __forceinline__ int cell_base_of_lane(const KernelArgs &k, int i, int lane) {
    return lane < 27 ? __ldg(k.cell_start + MLIP_CHECK_INDEX(neighbor_cell(k.grid, __ldg(k.cell_id + i), lane), k.grid.n_cells, k.status)) : 0;
}
template <int SCAN_CHUNKS, bool L16>
__device__ __forceinline__ int collect_pairs_n(const KernelArgs &k, const double4 &pi, int64_t beg, int64_t &cur, int64_t end, float4 *pq, int cap, int lane,
                                               const int *sidx, int n_pref, int cs) {
    int nq = 0;
    while (cur < end && nq + (int)min((int64_t)(SCAN_CHUNKS * 32), end - cur) <= cap) {
        int jj[SCAN_CHUNKS];
#pragma unroll
        for (int c = 0; c < SCAN_CHUNKS; ++c) {
            const int64_t e = cur + 32 * c + lane;
            if (L16) {   // (the prefetch copied whole 32-bit words starting at the even entry at or before `beg`)
                const int code = e < end ? (e - beg < n_pref ? reinterpret_cast<const uint16_t *>(sidx)[(e - beg) + (beg & 1)]
                                                             : __ldg(k.nbr16 + MLIP_CHECK_INDEX(e, k.nbr_cap, k.status))) : 0;
                const int base = __shfl_sync(0xffffffffu, cs, code >> L16_SHIFT);
                jj[c] = e < end ? base + (code & L16_MASK) : -1;
            } else {
                jj[c] = e < end ? (e - beg < n_pref ? sidx[e - beg] : __ldg(k.nbr + MLIP_CHECK_INDEX(e, k.nbr_cap, k.status))) : -1;
            }
            if (jj[c] >= 0) jj[c] = (int)MLIP_CHECK_INDEX(jj[c], k.n, k.status);
        }
        double4 pp[SCAN_CHUNKS];
#pragma unroll
        for (int c = 0; c < SCAN_CHUNKS; ++c) pp[c] = load_pos4(k.pos4 + (jj[c] < 0 ? 0 : jj[c]));
#pragma unroll
        for (int c = 0; c < SCAN_CHUNKS; ++c) {
            if (cur + 32 * c >= end) continue;   // warp-uniform: nothing in this chunk
            const double dx = min_image(pp[c].x - pi.x, k.grid.box[0], k.grid.half[0]);
            const double dy = min_image(pp[c].y - pi.y, k.grid.box[1], k.grid.half[1]);
            const double dz = min_image(pp[c].z - pi.z, k.grid.box[2], k.grid.half[2]);
            const double d2 = dx * dx + dy * dy + dz * dz;
            const bool valid = jj[c] >= 0 && d2 < k.rc2;
            const unsigned m = __ballot_sync(0xffffffffu, valid);
            if (valid)
                pq[nq + __popc(m & ((1u << lane) - 1u))] =
                    make_float4((float)dx, (float)dy, (float)dz, __int_as_float(jj[c] | ((int)pp[c].w << J_BITS)));
            nq += __popc(m);
        }
        cur += SCAN_CHUNKS * 32;
    }
    __syncwarp();
    return nq;
}
// Short lists (the usual case while the far entries are skipped) take the three-chunk form: fewer loads in flight,
// fewer registers.
template <bool L16>
__device__ __forceinline__ int collect_pairs(const KernelArgs &k, const double4 &pi, int64_t beg, int64_t &cur, int64_t end, float4 *pq, int cap, int lane,
                                             const int *sidx, int n_pref, int cs) {
    if (end - beg <= NARROW_CHUNKS * 32 || cap < WIDE_CHUNKS * 32) return collect_pairs_n<NARROW_CHUNKS, L16>(k, pi, beg, cur, end, pq, cap, lane, sidx, n_pref, cs);
    return collect_pairs_n<WIDE_CHUNKS, L16>(k, pi, beg, cur, end, pq, cap, lane, sidx, n_pref, cs);
}

// The pairs of a warp's two atoms, the second one's from the next multiple of sixteen on: the batches of 32 pairs in which the loops work
// then run over both (78 + 78 pairs are five of them, not three and three), and the gathers of both atoms are in flight together.  Lists of up
// to 96 entries each whose indices were prefetched (NextAtoms).  One evaluation in us, one atom after the other / side by side: 1,000,188 atoms
// of six species 7661 / 7466, 2,000,000 of the ionic solid (42 pairs) 11,367 / 10,726; 58 and 54 pairs, where no batch is saved, 432 / 434 and 1683 / 1687.
template <bool L16>
__device__ __forceinline__ void collect_two(const KernelArgs &k, const int *pf, int n_atoms, float4 *pq, int lane, int &n0, int &n1) {
    constexpr int CH = NARROW_CHUNKS;
    int jj[2][CH], len[2];
    double4 pi[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int *sidx = pf + u * PF_WORDS;
        len[u] = u < n_atoms ? sidx[PF_IDX + 3] : 0;
        const int odd = sidx[PF_IDX + 1] & 1;   // of the list's start (see stage_c)
        pi[u] = load_pos4(k.pos4 + (u < n_atoms ? sidx[PF_IDX] : 0));
        const int cs = L16 && lane < 27 ? sidx[PF_CS + lane] : 0;
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const int e = 32 * c + lane;
            if (L16) {
                const int code = e < len[u] ? reinterpret_cast<const uint16_t *>(sidx)[e + odd] : 0;
                const int base = __shfl_sync(0xffffffffu, cs, code >> L16_SHIFT);
                jj[u][c] = e < len[u] ? base + (code & L16_MASK) : -1;
            } else {
                jj[u][c] = e < len[u] ? sidx[e] : -1;
            }
            if (jj[u][c] >= 0) jj[u][c] = (int)MLIP_CHECK_INDEX(jj[u][c], k.n, k.status);
        }
    }
    double4 pp[2][CH];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int c = 0; c < CH; ++c) pp[u][c] = load_pos4(k.pos4 + (jj[u][c] < 0 ? 0 : jj[u][c]));
    int at = 0;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int first = at;
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            if (32 * c >= len[u]) continue;   // warp-uniform: nothing in this chunk
            const double dx = min_image(pp[u][c].x - pi[u].x, k.grid.box[0], k.grid.half[0]);
            const double dy = min_image(pp[u][c].y - pi[u].y, k.grid.box[1], k.grid.half[1]);
            const double dz = min_image(pp[u][c].z - pi[u].z, k.grid.box[2], k.grid.half[2]);
            const double d2 = dx * dx + dy * dy + dz * dz;
            const bool valid = jj[u][c] >= 0 && d2 < k.rc2;
            const unsigned m = __ballot_sync(0xffffffffu, valid);
            if (valid)
                pq[at + __popc(m & ((1u << lane) - 1u))] =
                    make_float4((float)dx, (float)dy, (float)dz, __int_as_float(jj[u][c] | ((int)pp[u][c].w << J_BITS)));
            at += __popc(m);
        }
        if (u == 0) { n0 = at; at = (at + 15) & ~15; }
        else n1 = at - first;
    }
    __syncwarp();
}
static_assert(2 * NARROW_CHUNKS * 32 <= Layout<2>::POOL, "two short lists fit the queue");

// ---------------- Encoding ----------------
// A lane's place in the encoding's k-steps: lane (g, t) evaluates chunk g (channels 4g ..) of pairs 2t, 2t + 1, 2t + 8, 2t + 9 of the
// k-step.  A pair in slot p takes its rows in the residue order p / 2, p / 2 + 1, .. (mod 4): the eight lanes of a load phase, two
// chunks of four pairs, then fall into eight bank groups.
struct EncodeLane {
    uint32_t chunk[2], a_addr;
    __device__ __forceinline__ EncodeLane(const float *stage, int lane) {
#pragma unroll
        for (int q = 0; q < 2; ++q) chunk[q] = 16u * ((lane >> 2) ^ table_swizzle(((lane & 3) + q) & 3));
        a_addr = smem_addr(stage) + ((lane & 7) + ((lane >> 4) << 3)) * (ST_STRIDE * 4) + ((lane >> 3) & 1) * 16;
    }
};
// Lane = pair: harmonics (Eq. 3) and spline basis of queue entry `slot` into the hand-over rows; zeros where there is no pair.
template <bool TAB_SMEM>
__device__ __forceinline__ void encode_rows(const KernelArgs &k, const TableView &tv, const float4 *pq, int slot, bool live, float *stage, int lane) {
    float h[D_ANG], b[4];
    int row = 0;
    if (live) {
        const float4 e = pq[slot];
        const float d2 = e.x * e.x + e.y * e.y + e.z * e.z, rinv = fast_rsqrt(d2), r = d2 * rinv;
        harmonics(e.x * rinv, e.y * rinv, e.z * rinv, h);
        float u;
        const int iv = spline_interval(r, k.tab.r_min, k.tab.inv_h, k.tab.knots, u, k.status);
        cubic_basis(u, b);
        row = (__float_as_int(e.w) >> J_BITS) * (k.tab.knots + 3) + iv;
    } else {
#pragma unroll
        for (int a = 0; a < D_ANG; ++a) h[a] = 0.f;
        b[0] = b[1] = b[2] = b[3] = 0.f;
    }
    uint32_t hi[8], lo[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) split_h2(h[2 * q], h[2 * q + 1], hi[q], lo[q]);
    uint4 *dst = reinterpret_cast<uint4 *>(stage + lane * ST_STRIDE);
    dst[0] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    dst[1] = make_uint4(hi[4], hi[5], hi[6], hi[7]);
    dst[2] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    dst[3] = make_uint4(lo[4], lo[5], lo[6], lo[7]);
    const int turn = ((lane >> 1) - row) & 3;
    *reinterpret_cast<float4 *>(dst + 4) = rotate4(b, turn);
    RowOffsets<TAB_SMEM> ro;
    ro.make(tv, row, turn);
    ro.store(stage + 32 * ST_STRIDE + lane * OFF_WORDS<TAB_SMEM>);
}
// Eq. 4 for the sixteen pairs of hand-over rows 16 ks .. (HALF: none behind the eighth, whose radial functions are not evaluated; with the
// derivation's half tiles and the sums over lanes by halves: 256,000 atoms of 54 pairs 1687 -> 1627 us an evaluation, the ionic solid 10,726 -> 10,362,
// six species 7466 -> 7458.  With one atom per warp the second form of the code cost 864 atoms 27 -> 29 us: not there.)
template <bool TAB_SMEM, bool HALF>
__device__ __forceinline__ void encode_kstep(const TableView &tv, const float *stage, const EncodeLane &el, int ks, int t, float (&Pf)[4][4]) {
    const float *offs = stage + 32 * ST_STRIDE;
    // A = H^T (16 x 16 pairs), stored pair by pair: transposed on the way in
    uint32_t ah[4], al[4];
    ldmatrix_x4_trans(ah, el.a_addr + ks * (16 * ST_STRIDE * 4));
    ldmatrix_x4_trans(al, el.a_addr + ks * (16 * ST_STRIDE * 4) + 32);
    // B = G (16 pairs x 8 channels per n-tile; column g of n-tile c is channel 4 g + c): g = sum_m b_m c_m (Eq. 2)
    uint32_t bh[4][2], bl[4][2];
    if (HALF) {
#pragma unroll
        for (int c = 0; c < 4; ++c) bh[c][1] = bl[c][1] = 0u;
    }
#pragma unroll
    for (int half = 0; half < (HALF ? 1 : 2); ++half) {
        float gv[2][4];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int slot = 16 * ks + 8 * half + 2 * t + u;
            const float4 b = *reinterpret_cast<const float4 *>(stage + slot * ST_STRIDE + 16);
            RowOffsets<TAB_SMEM> ro;
            ro.load(offs + slot * OFF_WORDS<TAB_SMEM>);
            const float bw[4] = {b.x, b.y, b.z, b.w};
            float2 lo = make_float2(0.f, 0.f), hi = lo;
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const float4 c = table_load<TAB_SMEM>(tv, ro.at(m, el.chunk));
                lo = ffma2(make_float2(bw[m], bw[m]), make_float2(c.x, c.y), lo);
                hi = ffma2(make_float2(bw[m], bw[m]), make_float2(c.z, c.w), hi);
            }
            gv[u][0] = lo.x; gv[u][1] = lo.y; gv[u][2] = hi.x; gv[u][3] = hi.y;
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) split_h2(gv[0][c], gv[1][c], bh[c][half], bl[c][half]);
    }
    // the three terms of each n-tile are issued interleaved over the n-tiles
    float c[4][4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) mma_f16_z(c[nt], al[0], al[1], al[2], al[3], bh[nt][0], bh[nt][1]);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) mma_f16(c[nt], ah[0], ah[1], ah[2], ah[3], bl[nt][0], bl[nt][1]);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) mma_f16(c[nt], ah[0], ah[1], ah[2], ah[3], bh[nt][0], bh[nt][1]);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const float2 s01 = add2(make_float2(Pf[nt][0], Pf[nt][1]), make_float2(c[nt][0], c[nt][1]));
        const float2 s23 = add2(make_float2(Pf[nt][2], Pf[nt][3]), make_float2(c[nt][2], c[nt][3]));
        Pf[nt][0] = s01.x; Pf[nt][1] = s01.y; Pf[nt][2] = s23.x; Pf[nt][3] = s23.y;
    }
}
__device__ __forceinline__ void clear_fragments(float (&Pf)[4][4]) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) Pf[a][b] = 0.f;
}

// One atom on its own: returns the number of pairs and the moment as accumulator fragments.
// `queued` returns the number of pairs left in the queue when the whole list fitted in one round
// (the derivation then reuses them), or -1.
// (UNROLL = 2, kernels without atoms side by side: two k-steps side by side and no half ones.  With one atom per warp the chain through a tile is the
// time; with two, 97,336 atoms of 158 pairs 1397 us an evaluation with half steps one by one, 1377 so.)
template <bool TAB_SMEM, bool L16, int UNROLL>
__device__ __forceinline__ int encode_atom(const KernelArgs &k, const TableView &tv, const double4 &pi, int64_t beg, int64_t end,
                                           float4 *pq, int cap, float *stage, int lane, float (&Pf)[4][4], int &queued, const int *sidx, int n_pref,
                                           int cs, PhaseClock &pc) {
    const EncodeLane el(stage, lane);
    clear_fragments(Pf);
    int total = 0, rounds = 0, n = 0;
    int64_t cur = beg;
    do {
        n = collect_pairs<L16>(k, pi, beg, cur, end, pq, cap, lane, sidx, n_pref, cs);
        pc.mark(0);
        for (int q0 = 0; q0 < n; q0 += 32) {
            encode_rows<TAB_SMEM>(k, tv, pq, q0 + lane, q0 + lane < n, stage, lane);
            __syncwarp();
            pc.mark(1);
#pragma unroll UNROLL
            for (int ks = 0; ks < 2; ++ks) {
                const int left = n - q0 - 16 * ks;
                if (left <= 0) break;
                if (UNROLL == 2 || left > 8) encode_kstep<TAB_SMEM, false>(tv, stage, el, ks, lane & 3, Pf);
                else encode_kstep<TAB_SMEM, true>(tv, stage, el, ks, lane & 3, Pf);
            }
            __syncwarp();
            pc.mark(2);
        }
        total += n;
        ++rounds;
    } while (cur < end);
    queued = rounds == 1 ? n : -1;
    return total;
}

// ---------------- Tensor memory (TMEM) ----------------
// The SM's 256 KB of tensor memory (128 lanes x 512 columns of 32 bits) is otherwise idle in this kernel (the
// contractions are per-atom products too small for tcgen05.mma), and it is the one on-chip store large enough for a
// species' head: 41 k weights in MMA-fragment order for the forward and the reverse pass, as fp16 hi + lo pairs (the layout
// is given at TM_FWD0 above).  A warp reaches the 32 lanes of quarter (warp % 4); all four warps of a quarter read the
// same 320 columns.  tcgen05.ld / st bypass the L1/shared-memory data pipe, which is this kernel's busiest unit.
constexpr uint32_t TM_COLS = 512;

__device__ __forceinline__ void tmem_st4(uint32_t addr, uint4 v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t addr, uint32_t (&r)[32]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                   "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
                   "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
                   "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(addr) : "memory");
}
// Accumulator fragments of a 16-pair tile -> 16 lanes x 32 columns: the 16x256b shape's register layout is the m16n8
// accumulator's, eight columns per n-tile.
__device__ __forceinline__ void tmem_st_vt(uint32_t addr, const float (&V)[2][4], const float (&T)[2][4]) {
    asm volatile("tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(addr),
                 "f"(V[0][0]), "f"(V[0][1]), "f"(V[0][2]), "f"(V[0][3]), "f"(V[1][0]), "f"(V[1][1]), "f"(V[1][2]), "f"(V[1][3]),
                 "f"(T[0][0]), "f"(T[0][1]), "f"(T[0][2]), "f"(T[0][3]), "f"(T[1][0]), "f"(T[1][1]), "f"(T[1][2]), "f"(T[1][3]) : "memory");
}
// 16 registers of every lane to / from 16 columns (the moment P between encoding and derivation)
__device__ __forceinline__ void tmem_st16(uint32_t addr, const float (&P)[4][4]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(addr),
                 "f"(P[0][0]), "f"(P[0][1]), "f"(P[0][2]), "f"(P[0][3]), "f"(P[1][0]), "f"(P[1][1]), "f"(P[1][2]), "f"(P[1][3]),
                 "f"(P[2][0]), "f"(P[2][1]), "f"(P[2][2]), "f"(P[2][3]), "f"(P[3][0]), "f"(P[3][1]), "f"(P[3][2]), "f"(P[3][3]) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&P)[4][4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=f"(P[0][0]), "=f"(P[0][1]), "=f"(P[0][2]), "=f"(P[0][3]), "=f"(P[1][0]), "=f"(P[1][1]), "=f"(P[1][2]), "=f"(P[1][3]),
                   "=f"(P[2][0]), "=f"(P[2][1]), "=f"(P[2][2]), "=f"(P[2][3]), "=f"(P[3][0]), "=f"(P[3][1]), "=f"(P[3][2]), "=f"(P[3][3])
                 : "r"(addr) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// A warp copies its fourth of its quarter's weight columns for the species whose packed weights start at hp (ten 16-byte
// loads in flight at a time: a small system's kernel time is made of such round trips).
__device__ __forceinline__ void tmem_fill(uint32_t quarter_base, const uint32_t *__restrict__ hp, int warp, int lane) {
    constexpr int VECS = TM_VT / 4 / (NW / 4), STEP = 10;   // 16-byte vectors per lane and warp
    static_assert(VECS % STEP == 0 && NW % 4 == 0, "weight columns divide evenly over the warps of a quarter");
    const int v0 = (warp >> 2) * VECS;
    const uint4 *src = reinterpret_cast<const uint4 *>(hp) + ((size_t)(warp & 3) * (TM_VT / 4) + v0) * 32 + lane;
#pragma unroll
    for (int v = 0; v < VECS; v += STEP) {
        uint4 r[STEP];
#pragma unroll
        for (int q = 0; q < STEP; ++q) r[q] = __ldg(src + (size_t)(v + q) * 32);
#pragma unroll
        for (int q = 0; q < STEP; ++q) tmem_st4(quarter_base + 4 * (v0 + v + q), r[q]);
    }
    tmem_wait_st();
}

// ---------------- Derivation (Eq. 8-10) ----------------
// Lane = pair: spline basis and its derivative of queue entry `slot` into the hand-over rows; zeros where there is no pair.
template <bool TAB_SMEM>
__device__ __forceinline__ void derive_rows(const KernelArgs &k, const TableView &tv, const float4 *pq, int slot, bool live, float *bs, int lane) {
    float b[4] = {0.f, 0.f, 0.f, 0.f}, db[4] = {0.f, 0.f, 0.f, 0.f};
    int row = 0;
    if (live) {
        const float4 ent = pq[slot];
        const float d2 = ent.x * ent.x + ent.y * ent.y + ent.z * ent.z, r = d2 * fast_rsqrt(d2);
        float u;
        const int iv = spline_interval(r, k.tab.r_min, k.tab.inv_h, k.tab.knots, u, k.status);
        cubic_basis(u, b);
        cubic_basis_deriv(u, 1.f, db);
        row = (__float_as_int(ent.w) >> J_BITS) * (k.tab.knots + 3) + iv;
    }
    const int turn = (lane - row) & 3;
    float *dst = bs + lane * BS_STRIDE;
    *reinterpret_cast<float4 *>(dst) = rotate4(b, turn);
    *reinterpret_cast<float4 *>(dst + 4) = rotate4(db, turn);
    RowOffsets<TAB_SMEM> ro;
    ro.make(tv, row, turn);
    ro.store(dst + 8);
}
// W_i = dE_i/dP_i as B fragments of W_i^T times 1 / inv; k-step q holds channels 8t + 4q .. + 3 of lane (g, t).
struct WFragments {
    uint32_t hi[2][2][2], lo[2][2][2];   // [k-step][n-tile][b0, b1]
};
// V and T of the sixteen pairs of hand-over rows 16 mt .. to tensor memory.  Tile fragments: lane (g, t) evaluates chunks 2t, 2t + 1 of pairs
// g, g + 8.  A pair in slot p takes its rows in the residue order p, p + 1, .. (mod 4): of the two pairs in a load phase one reads the
// even, the other the odd chunk positions.  HALF: no pair behind the eighth.
template <bool TAB_SMEM, bool HALF>
__device__ __forceinline__ void derive_tile(const TableView &tv, const float *bs, int mt, int g, const uint32_t (&chunk)[2], const WFragments &W, uint32_t tm_vt) {
    // A = [G; G'] (16 pairs x 32 channels): rows pairs g, g + 8; this lane evaluates channels 8t .. 8t+7
    // (one accumulator per output here: the truncating accumulation costs ~1e-6 relative on a
    // short chain, irrelevant for forces, and the registers are needed elsewhere).  G' is the derivative per knot interval.
    float V[2][4], T[2][4];
    uint32_t ah[2][4], al[2][4], dh[2][4], dl[2][4];   // [k-step][fragment register]
    if (HALF) {
#pragma unroll
        for (int ks = 0; ks < 2; ++ks)
#pragma unroll
            for (int r = 1; r < 4; r += 2) ah[ks][r] = al[ks][r] = dh[ks][r] = dl[ks][r] = 0u;
    }
#pragma unroll
    for (int q = 0; q < (HALF ? 1 : 2); ++q) {
        const float *rp = bs + (16 * mt + g + 8 * q) * BS_STRIDE;
        const float4 b = *reinterpret_cast<const float4 *>(rp), db = *reinterpret_cast<const float4 *>(rp + 4);
        RowOffsets<TAB_SMEM> ro;
        ro.load(rp + 8);
        const float bw[4] = {b.x, b.y, b.z, b.w}, dbw[4] = {db.x, db.y, db.z, db.w};
        float2 G2[4], dG2[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) { G2[c] = make_float2(0.f, 0.f); dG2[c] = make_float2(0.f, 0.f); }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const uint32_t at = ro.at(m, chunk);
            const float4 c0 = table_load<TAB_SMEM>(tv, at), c1 = table_load<TAB_SMEM>(tv, at ^ 16u);
            const float2 cv[4] = {make_float2(c0.x, c0.y), make_float2(c0.z, c0.w), make_float2(c1.x, c1.y), make_float2(c1.z, c1.w)};
            const float2 b2 = make_float2(bw[m], bw[m]), db2 = make_float2(dbw[m], dbw[m]);
#pragma unroll
            for (int c = 0; c < 4; ++c) { G2[c] = ffma2(b2, cv[c], G2[c]); dG2[c] = ffma2(db2, cv[c], dG2[c]); }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {   // channel pair c: k-step c / 2, fragment register q + 2 (c % 2)
            split_h2(G2[c].x, G2[c].y, ah[c >> 1][q + 2 * (c & 1)], al[c >> 1][q + 2 * (c & 1)]);
            split_h2(dG2[c].x, dG2[c].y, dh[c >> 1][q + 2 * (c & 1)], dl[c >> 1][q + 2 * (c & 1)]);
        }
    }
    // Eq. 9 (rows of V: a = 0..7 and 8..15) and W g' (Eq. 8 re-associated); cross terms first, the four
    // independent accumulators interleaved
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            if (ks == 0) {
                mma_f16_z(V[nt], al[ks][0], al[ks][1], al[ks][2], al[ks][3], W.hi[ks][nt][0], W.hi[ks][nt][1]);
                mma_f16_z(T[nt], dl[ks][0], dl[ks][1], dl[ks][2], dl[ks][3], W.hi[ks][nt][0], W.hi[ks][nt][1]);
            } else {
                mma_f16(V[nt], al[ks][0], al[ks][1], al[ks][2], al[ks][3], W.hi[ks][nt][0], W.hi[ks][nt][1]);
                mma_f16(T[nt], dl[ks][0], dl[ks][1], dl[ks][2], dl[ks][3], W.hi[ks][nt][0], W.hi[ks][nt][1]);
            }
        }
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            mma_f16(V[nt], ah[ks][0], ah[ks][1], ah[ks][2], ah[ks][3], W.lo[ks][nt][0], W.lo[ks][nt][1]);
            mma_f16(T[nt], dh[ks][0], dh[ks][1], dh[ks][2], dh[ks][3], W.lo[ks][nt][0], W.lo[ks][nt][1]);
        }
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            mma_f16(V[nt], ah[ks][0], ah[ks][1], ah[ks][2], ah[ks][3], W.hi[ks][nt][0], W.hi[ks][nt][1]);
            mma_f16(T[nt], dh[ks][0], dh[ks][1], dh[ks][2], dh[ks][3], W.hi[ks][nt][0], W.hi[ks][nt][1]);
        }
    }
    // The accumulator fragments of the 16 pairs go to tensor memory as 16 lanes (pair) x 32 columns (V, T); read back
    // with lane = pair.  (Through shared memory the same exchange was 188 of the kernel's 1,958 L1 wavefronts per atom.)
    tmem_st_vt(tm_vt + ((uint32_t)(16 * mt) << 16), V, T);
}
// Lane = pair: projection onto the pair vector (Eq. 10), scatter of the reaction; returns the force on the central atom.
template <bool DET>
__device__ __forceinline__ float3 project_pair(const KernelArgs &k, const float4 &ent, const uint32_t (&vt)[32], float w_scale_inv, float (&vir)[9]) {
    float v[D_ANG], tt[D_ANG];
#pragma unroll
    for (int q = 0; q < D_ANG; ++q) { v[q] = __uint_as_float(vt[q]); tt[q] = __uint_as_float(vt[16 + q]); }
    const float x = ent.x, y = ent.y, z = ent.z;
    const float rinv = fast_rsqrt(x * x + y * y + z * z);
    const int j = __float_as_int(ent.w) & ((1 << J_BITS) - 1);
    const float ux = x * rinv, uy = y * rinv, uz = z * rinv;
    float s, tx, ty, tz, tu;
    harmonics_project(ux, uy, uz, v, tt, s, tx, ty, tz, tu);
    // f_ij = (g' . u_ij) r^ + J_ang^T v_ij,  J_ang = (grad_u h)(I - u u^T) / r, the scales taken back
    const float sr = s * (w_scale_inv * k.tab.inv_h), vr = rinv * w_scale_inv;
    const float qx = sr * ux + (tx - tu * ux) * vr;
    const float qy = sr * uy + (ty - tu * uy) * vr;
    const float qz = sr * uz + (tz - tu * uz) * vr;
    if (DET) fixed_add3(k.force_fx + 3 * (size_t)j, -qx, -qy, -qz);
    else atomicAdd(&k.force[j], make_float4(-qx, -qy, -qz, 0.f));   // one 128-bit reduction per pair
    vir[0] -= x * qx; vir[1] -= x * qy; vir[2] -= x * qz;
    vir[3] -= y * qx; vir[4] -= y * qy; vir[5] -= y * qz;
    vir[6] -= z * qx; vir[7] -= z * qy; vir[8] -= z * qz;
    return make_float3(qx, qy, qz);
}
// The sum over the lanes, each step sending what the lane does not keep: six shuffles (they use the shared-memory pipe) instead of fifteen.
template <bool DET>
__device__ __forceinline__ void add_own_force(const KernelArgs &k, int i, float3 f, int lane) {
    const bool upper = lane & 16, odd = lane & 8;
    float p = upper ? f.z : f.x, q = upper ? 0.f : f.y;
    p += __shfl_xor_sync(0xffffffffu, upper ? f.x : f.z, 16);
    q += __shfl_xor_sync(0xffffffffu, upper ? f.y : 0.f, 16);
    float v = (odd ? q : p) + __shfl_xor_sync(0xffffffffu, odd ? p : q, 8);
#pragma unroll
    for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((lane & 7) == 0 && lane < 24) {   // lanes 0, 8, 16: x, y, z
        if (DET) atomicAdd(reinterpret_cast<unsigned long long *>(k.force_fx + 3 * (size_t)i + (lane >> 3)), (unsigned long long)__float2ll_rn(v * FORCE_FX));
        else atomicAdd(&k.force[i].x + (lane >> 3), v);
    }
}
__device__ __forceinline__ void derive_chunks(uint32_t (&chunk)[2], int lane) {
#pragma unroll
    for (int q = 0; q < 2; ++q) chunk[q] = 16u * ((2 * (lane & 3)) ^ table_swizzle(((lane >> 2) + q) & 3));
}

// One atom on its own.
template <bool SIDE, bool TAB_SMEM, bool DET, bool L16>
__device__ __forceinline__ void derive_atom(const KernelArgs &k, const TableView &tv, int i,
                                            float4 *pq, int cap, float *scr, int queued, int lane, const WFragments &W, float w_scale_inv,
                                            float (&vir)[9], uint32_t tm_vt, PhaseClock &pc) {
    uint32_t chunk[2];
    derive_chunks(chunk, lane);
    float3 f = make_float3(0.f, 0.f, 0.f);

    auto batch = [&](int first, int n) {
        derive_rows<TAB_SMEM>(k, tv, pq, first + lane, lane < n, scr, lane);
        __syncwarp();
        pc.mark(4);
        const int nmt = (n + 15) >> 4;
#pragma unroll 1
        for (int mt = 0; mt < nmt; ++mt) {
            if (!SIDE || n - 16 * mt > 8) derive_tile<TAB_SMEM, false>(tv, scr, mt, lane >> 2, chunk, W, tm_vt);
            else derive_tile<TAB_SMEM, true>(tv, scr, mt, lane >> 2, chunk, W, tm_vt);
        }
        tmem_wait_st();
        pc.mark(5);
        uint32_t vt[32];
        tmem_ld32(tm_vt, vt);
        tmem_wait_ld();
        if (lane < n) {
            const float3 q = project_pair<DET>(k, pq[first + lane], vt, w_scale_inv, vir);
            f.x += q.x; f.y += q.y; f.z += q.z;
        }
        __syncwarp();
        pc.mark(6);
    };
    if (queued >= 0) {   // the encoding left every pair of this atom in the queue
        for (int q0 = 0; q0 < queued; q0 += 32) batch(q0, min(32, queued - q0));
    } else {   // rare: the list did not fit the queue; position and list bounds are fetched again rather than kept
               // in registers through the head
        const double4 pi = load_pos4(k.pos4 + i);
        const int64_t beg = k.nbr_off[i], end = *k.far_flag ? k.nbr_off[i + 1] : beg + k.nbr_near[i];
        int64_t cur = beg;
        const int cs = L16 ? cell_base_of_lane(k, i, lane) : 0;
        do {
            const int n = collect_pairs<L16>(k, pi, beg, cur, end, pq, cap, lane, nullptr, 0, cs);
            pc.mark(3);
            for (int q0 = 0; q0 < n; q0 += 32) batch(q0, min(32, n - q0));
        } while (cur < end);
    }
    add_own_force<DET>(k, i, f, lane);
}

// Barrier among the 256 threads of one group (hardware barrier 1 + group).
__device__ __forceinline__ void group_sync(int group) {
    asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "r"(GW * 32) : "memory");
}

// Head contraction on the tensor pipe: C^T[16 rows of W x 8 atoms] over four 16-wide k-steps.  A = wr (32 columns of tensor
// memory), B = activations in fragment order from shared memory; every k-step gets its own accumulator (four independent
// chains of three products), summed in fp32.  SCALED: `inv` holds the k-steps' scales of the lane's two atoms (act_store_scaled).
template <bool SCALED>
__device__ __forceinline__ void head_gemm(float (&c)[4], const uint32_t (&wr)[32], const uint4 *__restrict__ act, const uint32_t *inv = nullptr) {
    float acc[4][4];
    uint4 b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) b[u] = act[32 * u];
#pragma unroll
    for (int u = 0; u < 4; ++u) mma_f16_z(acc[u], wr[8 * u + 4], wr[8 * u + 5], wr[8 * u + 6], wr[8 * u + 7], b[u].x, b[u].z);
#pragma unroll
    for (int u = 0; u < 4; ++u) mma_f16(acc[u], wr[8 * u], wr[8 * u + 1], wr[8 * u + 2], wr[8 * u + 3], b[u].y, b[u].w);
#pragma unroll
    for (int u = 0; u < 4; ++u) mma_f16(acc[u], wr[8 * u], wr[8 * u + 1], wr[8 * u + 2], wr[8 * u + 3], b[u].x, b[u].z);
    if (!SCALED) {
#pragma unroll
        for (int e = 0; e < 4; ++e) c[e] = (acc[0][e] + acc[1][e]) + (acc[2][e] + acc[3][e]);
        return;
    }
    const uint4 w = *reinterpret_cast<const uint4 *>(inv);
    const float2 s[4] = {unpack_bf16(w.x), unpack_bf16(w.y), unpack_bf16(w.z), unpack_bf16(w.w)};
#pragma unroll
    for (int e = 0; e < 4; e += 2) {
        float2 sum = make_float2(acc[0][e] * s[0].x, acc[0][e + 1] * s[0].y);
#pragma unroll
        for (int u = 1; u < 4; ++u) sum = ffma2(make_float2(acc[u][e], acc[u][e + 1]), s[u], sum);
        c[e] = sum.x; c[e + 1] = sum.y;
    }
}

// Activations in B-fragment order.  k-step s covers neurons (or inputs) 16 s .. 16 s + 15, its k-index 2 j + h standing for
// neuron 16 s + j + 8 h, so that the two values a lane of an accumulator fragment holds for one atom (neurons g, g + 8) are one
// fp16 pair.  Fragment lane (atom a, quad lane q) reads {pair q, pair q + 4}; atom rows are stored in the order
// act_row(a), which spreads a store over all banks.
__device__ __forceinline__ int act_row(int a) { return (a & 4) | ((a & 1) << 1) | ((a >> 1) & 1); }
__device__ __forceinline__ void act_store(float *act, int kstep, int atom, int j, uint32_t hi, uint32_t lo) {
    *reinterpret_cast<uint2 *>(act + kstep * ACT_KSTEP + (act_row(atom) * 4 + (j & 3)) * 4 + 2 * (j >> 2)) = make_uint2(hi, lo);
}

// One warp's 16 neurons (m-tile mt) of the lane's atoms, values {n0 a, n0 a+1, n1 a, n1 a+1}, as the next contraction's k-step: scaled by the
// power of two that brings the largest of an atom's 16 values just below 2^15, the inverse (bf16 pairs [atom pair][k-step]) beside them.
// Measured, not taken from the weights' norms: a product over the layers of row or column sums of large weights lies so far above the
// values that the lower halves, and with them the forces' digits, were lost (hidden layers x 300 with small pre-activations: 8e-2
// relative, now 1e-6).  Three shuffles in the chain from layer to layer, a store and a 16-byte load per contraction: an evaluation of 5,544
// atoms 61.8 -> 63.3 us, 65,536 atoms NVE 4924 -> 5013 us per 10 steps, 8,001,504 atoms 683.8 -> 691.5 ms.
__device__ __forceinline__ void act_store_scaled(float *act, uint32_t *inv, int mt, int atom, int g, int t, const float (&m)[4]) {
    const float b0 = fmaxf(fabsf(m[0]), fabsf(m[2])), b1 = fmaxf(fabsf(m[1]), fabsf(m[3]));
    uint32_t most = __byte_perm(__float_as_uint(b0), __float_as_uint(b1), 0x7632);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) most = __vmaxu2(most, __shfl_xor_sync(0xffffffffu, most, o));
    const uint32_t w = inverse_scales(most);
    if (g == 0) inv[(atom >> 1) * (HEAD_H / 16) + mt] = w;
    const float2 s = unpack_bf16(inverse_of(w));
    uint32_t hi, lo;
    split_h2(m[0] * s.x, m[2] * s.x, hi, lo);
    act_store(act, mt, 2 * t, g, hi, lo);
    split_h2(m[1] * s.y, m[3] * s.y, hi, lo);
    act_store(act, mt, 2 * t + 1, g, hi, lo);
}

// Prefetch of the warp's atoms in the group's NEXT tile, spread over three points of the head so
// that each dependent global load has a barrier's worth of time to arrive: centre index -> list
// bounds (lane u for the warp's u-th atom) -> the first PF_IDX neighbor indices (cp.async straight into shared memory).
// (Pulling the neighbors' positions into L2 as a fourth step cost more issue slots than it saved latency.)
template <int APW>
struct NextAtoms {
    const KernelArgs *k;
    int *pf;          // shared: per atom PF_IDX neighbor indices, then {atom, list start lo, list start hi, list length}
    int slot;         // lane u < APW: position in center_order, or -1
    int i;
    bool use_far;     // the lists' far entries have to be scanned as well
    int64_t beg;
    int len;
    int cid;          // compact lists: the atom's build-time cell
    __device__ __forceinline__ void stage_a() { if (slot >= 0) i = (int)MLIP_CHECK_INDEX(__ldg(k->center_order + MLIP_CHECK_INDEX(slot, k->n, k->status)), k->n, k->status); }
    template <bool L16>
    __device__ __forceinline__ void stage_b() {
        if (slot >= 0) {
            beg = __ldg(k->nbr_off + i);
            len = use_far ? (int)(__ldg(k->nbr_off + i + 1) - beg) : __ldg(k->nbr_near + i);
            if (L16) cid = __ldg(k->cell_id + i);
        }
    }
    template <bool L16>
    __device__ __forceinline__ void stage_c(int lane) {
#pragma unroll
        for (int u = 0; u < APW; ++u) {
            if (__shfl_sync(0xffffffffu, slot, u) < 0) break;   // (a ragged tile's atoms come first)
            int *sidx = pf + u * PF_WORDS;
            const int64_t b = __shfl_sync(0xffffffffu, beg, u);
            const int n = min(PF_IDX, __shfl_sync(0xffffffffu, len, u));
            if (L16) {   // codes travel as whole 32-bit words from the even entry at or before `b`; the 27 cell bases follow them
                const int cell = __shfl_sync(0xffffffffu, cid, u);
                const int odd = (int)(b & 1), words = (odd + n + 1) >> 1;
                const int *src = reinterpret_cast<const int *>(k->nbr16 + (b - odd));
#pragma unroll
                for (int c = 0; c < (PF_IDX / 2 + 1 + 31) / 32; ++c) {
                    const int e = 32 * c + lane;
                    if (e < words) {
                        const int at = MLIP_CHECK_INDEX(b - odd + 2 * e, k->nbr_cap, k->status) == b - odd + 2 * e ? e : 0;
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(sidx + e)), "l"(src + at) : "memory");
                    }
                }
                if (lane < 27)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(sidx + PF_CS + lane)),
                                 "l"(k->cell_start + MLIP_CHECK_INDEX(neighbor_cell(k->grid, cell, lane), k->grid.n_cells, k->status)) : "memory");
            } else {
#pragma unroll
                for (int c = 0; c < PF_IDX / 32; ++c) {
                    const int e = 32 * c + lane;
                    if (e < n) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(sidx + e)), "l"(k->nbr + MLIP_CHECK_INDEX(b + e, k->nbr_cap, k->status)) : "memory");
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (lane < APW && slot >= 0) {
            int *meta = pf + lane * PF_WORDS + PF_IDX;
            meta[0] = i; meta[1] = (int)(beg & 0xffffffff); meta[2] = (int)(beg >> 32); meta[3] = len;
        }
    }
};

// ---------------- Regression (Eq. 6) forward and reverse for the group's tile ----------------
// One atom's invariants (warp = atom) -> scaled fp16 pairs in fragment order, and sc[atom] = the factor that takes the first layer's
// product back.
__device__ __forceinline__ void split_invariants(const float *xrow, float *xs, float *sc, const float *hc, int atom, int lane) {
    xs += (atom >> 3) * XS_WORDS;
    // lane handles the pairs (c, c + 8) number lane and lane + 32 of the 64: k-step p / 8, j = p % 8
    const int j = lane & 7, s0 = lane >> 3, s1 = s0 + 4;
    const float *cs = hc + HC_CS;
    const float a0 = xrow[16 * s0 + j] * cs[16 * s0 + j], a1 = xrow[16 * s0 + 8 + j] * cs[16 * s0 + 8 + j];
    const float b0 = xrow[16 * s1 + j] * cs[16 * s1 + j], b1 = xrow[16 * s1 + 8 + j] * cs[16 * s1 + 8 + j];
    const float most = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(fmaxf(fabsf(a0), fabsf(a1)), fmaxf(fabsf(b0), fabsf(b1))))));
    const float sx = scale_for(most);
    uint32_t hi, lo;
    split_h2(a0 * sx, a1 * sx, hi, lo);
    act_store(xs, s0, atom & 7, j, hi, lo);
    split_h2(b0 * sx, b1 * sx, hi, lo);
    act_store(xs, s1, atom & 7, j, hi, lo);
    if (lane == 0) sc[atom] = inverse_pow2(sx) * hc[HC_WS];
}

// In: xs = split invariants.  Out: sX = dE/dG [atom][128]; per-atom energies written.  wg = warp within the group: it owns
// m-tile wg % 4 (16 neurons) of the atoms 8 (wg / 4) .. + 7 through all layers (one atom per warp: warps 4..7 own nothing).
template <int APW, bool DET, bool L16>
__device__ __forceinline__ void head_tile(const KernelArgs &k, const float *xs, float *sX, const float *sc, uint32_t *us, float *ep, float *zs, const float *hc,
                                          uint32_t tm, int count, int first, int group, int wg, int lane, double &e_sum, NextAtoms<APW> &nx, PhaseClock &pc) {
    constexpr int NA = GW * APW;
    const int g = lane >> 2, t = lane & 3, mt = wg & 3, nt = wg >> 2;
    const int frag = act_row(g) * 4 + t;        // this lane's vector of a k-step
    const bool owner = APW == 2 || wg < 4;
    const int a0 = (APW == 2 ? 8 * nt : 0) + 2 * t;   // the lane's atoms: a0, a0 + 1
    const int n0 = 16 * mt + g, n1 = n0 + 8;    // and neurons: its values are {n0 a0, n0 a0+1, n1 a0, n1 a0+1}
    constexpr int US = Layout<APW>::US;
    const uint32_t *my_us = us + (a0 >> 1) * (HEAD_H / 16);   // the lane's atoms' activation scales, of a layer in buffer 0
    if (APW == 2) { xs += nt * XS_WORDS; zs += nt * 2 * ZS_WORDS; }
    float y[4] = {0.f, 0.f, 0.f, 0.f};          // running activations (the skip path)
    float dz[4];                                // dE/dy in the reverse pass
    float sd[HEAD_L][4];                        // SiLU' of the pre-activations, layer by layer
    uint32_t w[32];                             // A fragments of the coming contraction
#pragma unroll
    for (int L = 0; L < HEAD_L; ++L) {
        const float *zin = zs + ((L + 1) & 1) * ZS_WORDS;
        float *zout = zs + (L & 1) * ZS_WORDS;
        if (owner) {
            float c[4];
            tmem_ld32(tm + (L == 0 ? TM_FWD0 : TM_FWD + 32 * (L - 1)), w);
            tmem_wait_ld();
            float2 u = make_float2(hc[HC_WS + L], hc[HC_WS + L]);
            if (L == 0) {
                float c2[4];
                head_gemm<false>(c, w, reinterpret_cast<const uint4 *>(xs) + frag);
                tmem_ld32(tm + TM_FWD0 + 32, w);
                tmem_wait_ld();
                head_gemm<false>(c2, w, reinterpret_cast<const uint4 *>(xs + 4 * ACT_KSTEP) + frag);
#pragma unroll
                for (int e = 0; e < 4; ++e) c[e] += c2[e];
                u = *reinterpret_cast<const float2 *>(sc + a0);
            } else {
                head_gemm<true>(c, w, reinterpret_cast<const uint4 *>(zin) + frag, my_us + ((L + 1) & 1) * US);
            }
            pc.mark(12);
            const float bias0 = hc[L * HEAD_H + n0], bias1 = hc[L * HEAD_H + n1];
            y[0] += silu_f(c[0] * u.x + bias0, sd[L][0]); y[1] += silu_f(c[1] * u.y + bias0, sd[L][1]);
            y[2] += silu_f(c[2] * u.x + bias1, sd[L][2]); y[3] += silu_f(c[3] * u.y + bias1, sd[L][3]);
            float m[4] = {y[0], y[1], y[2], y[3]};   // what goes to the next contraction
            if (L == HEAD_L - 1) {   // output layer and the start of the reverse pass: dE/dy = w_out
                const float wo0 = hc[HC_WOUT + n0], wo1 = hc[HC_WOUT + n1];
                float e0 = wo0 * y[0] + wo1 * y[2], e1 = wo0 * y[1] + wo1 * y[3];
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) {
                    e0 += __shfl_xor_sync(0xffffffffu, e0, o);
                    e1 += __shfl_xor_sync(0xffffffffu, e1, o);
                }
                if (g == 0) *reinterpret_cast<float2 *>(ep + mt * NA + a0) = make_float2(e0, e1);
                dz[0] = dz[1] = wo0; dz[2] = dz[3] = wo1;
#pragma unroll
                for (int e = 0; e < 4; ++e) m[e] = dz[e] * sd[L][e];
            }
            act_store_scaled(zout, us + (L & 1) * US, mt, a0, g, t, m);
        }
        if (L == 0) nx.stage_a();
        if (L == 1) nx.template stage_b<L16>();
        if (L == 2) nx.template stage_c<L16>(lane);
        pc.mark(13);
        group_sync(group);
        pc.mark(14);
    }
    if (wg == 7 && lane < count) {
        const float e_i = ((ep[lane] + ep[NA + lane]) + (ep[2 * NA + lane] + ep[3 * NA + lane])) + hc[HC_BOUT];
        k.e_atom[MLIP_CHECK_INDEX(__ldg(k.center_order + first + lane), k.n, k.status)] = e_i;
        e_sum += DET ? rint((double)e_i * ENERGY_FX) : (double)e_i;   // DET: exact integer sums
    }

    // reverse through the hidden layers 3, 2, 1 (each with its skip path); dE/dpre_3 sits where layer 3 put it
#pragma unroll
    for (int L = HEAD_L - 1; L >= 1; --L) {
        const float *zin = zs + (L & 1) * ZS_WORDS;
        float *zout = zs + ((L + 1) & 1) * ZS_WORDS;
        if (owner) {
            float c[4];
            tmem_ld32(tm + TM_BWD + 32 * (L - 1), w);
            tmem_wait_ld();
            head_gemm<true>(c, w, reinterpret_cast<const uint4 *>(zin) + frag, my_us + (L & 1) * US);
            const float u = hc[HC_WS + L];
            float m[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) { dz[e] += c[e] * u; m[e] = dz[e] * sd[L - 1][e]; }
            act_store_scaled(zout, us + ((L + 1) & 1) * US, mt, a0, g, t, m);
        }
        group_sync(group);
    }
    // first layer: dE/dG [128 x atoms], 16 inputs per m-tile: the warp's m-tiles mt, mt + 4 (one atom per warp: m-tile wg)
#pragma unroll
    for (int h = 0; h < APW; ++h) {
        const int m = APW == 2 ? mt + 4 * h : wg;
        float c[4];
        tmem_ld32(tm + TM_BWD0 + 32 * (m >> 2), w);
        tmem_wait_ld();
        head_gemm<true>(c, w, reinterpret_cast<const uint4 *>(zs) + frag, my_us);   // layer 0's dE/dpre: buffer 0
        const float u = hc[HC_WS], ua = u * hc[HC_CS + 16 * m + g], ub = u * hc[HC_CS + 16 * m + g + 8];
        float *p = sX + a0 * X_STRIDE + 16 * m + g;
        p[0] = c[0] * ua; p[X_STRIDE] = c[1] * ua; p[8] = c[2] * ub; p[X_STRIDE + 8] = c[3] * ub;
    }
    group_sync(group);
}

constexpr int TOTALS = 9 + 16 + 1;   // per warp at the end: virial, E_i sums of up to 16 lanes, pairs
// SIDE: a warp's two atoms go through the pair loops side by side where their pairs fit its queue together.
template <int APW, bool SIDE, bool TAB_SMEM, bool DET, bool L16>
__global__ void __launch_bounds__(NW * 32, 1) k_mega(const __grid_constant__ KernelArgs k, int tab_words) {
    static_assert(APW == 2 || !SIDE, "two atoms side by side");
    extern __shared__ __align__(128) float smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    using LY = Layout<APW>;
    constexpr int NA = LY::NA;
    const int group = warp / GW, wg = warp % GW;
    const int g = lane >> 2, t = lane & 3;
    float *s_tab = smem;                                   // [C][rows][K_RADIAL] when TAB_SMEM
    float *xs = smem + (TAB_SMEM ? tab_words : 0) + group * LY::GROUP;
    float *sX = xs + APW * XS_WORDS, *sc = sX + LY::SX + 2 * LY::US, *ep = sc + NA;
    uint32_t *us = reinterpret_cast<uint32_t *>(sX + LY::SX);
    float *scr_all = smem + (TAB_SMEM ? tab_words : 0) + NG * LY::GROUP;
    float *zs = scr_all + group * GW * SCR_WORDS;          // layer activations = the scratch of the group's warps
    float *scr = scr_all + warp * SCR_WORDS;
    float4 *pq = reinterpret_cast<float4 *>(scr_all + NW * SCR_WORDS + warp * LY::Q_WORDS);
    int *pf = reinterpret_cast<int *>(scr_all + NW * (SCR_WORDS + LY::Q_WORDS)) + warp * APW * PF_WORDS;
    int *info = reinterpret_cast<int *>(scr_all + NW * (SCR_WORDS + LY::Q_WORDS + APW * PF_WORDS)) + warp * LY::INFO;
    float *hc = scr_all + NW * LY::WARP;
    int *ctl = reinterpret_cast<int *>(hc + HC_WORDS);
    const int rows = k.tab.knots + 3;
    allow_next();
    if (!k.early) stamp_begin(k.stamp);   // (else from the end of the kernel ahead, whose time hides the staging)

    // all of tensor memory (this is the only CTA on the SM) for the head's weights
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(ctl + 4)), "r"(TM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();
    const uint32_t tm_base = *reinterpret_cast<volatile uint32_t *>(ctl + 4);
    const uint32_t tm_quarter = tm_base + ((uint32_t)(32 * (warp & 3)) << 16);
    const uint32_t tm_vt = tm_quarter + TM_VT + 32 * (warp >> 2), tm_p = tm_quarter + TM_P + 16 * (warp >> 2);

    double e_sum = 0.0;
    float vir[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    double vir_fx = 0.0;   // DET: lane q < 9 keeps component q as an exact integer-valued sum
    unsigned long long n_pairs = 0;
    TableView tv;
    PhaseClock pc;
    pc.start();

    // the tables and weights of a species
    auto stage = [&](int species) {
        const float *tab = k.tab.coef + (size_t)species * k.n_species * rows * K_RADIAL;
        if (TAB_SMEM) {
            const float4 *src = reinterpret_cast<const float4 *>(tab);
            const int n4 = k.n_species * rows * (K_RADIAL / 4);
#pragma unroll 4
            for (int idx = threadIdx.x; idx < n4; idx += NW * 32)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(reinterpret_cast<float4 *>(s_tab) + idx)), "l"(src + idx) : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
            tv.base = s_tab; tv.saddr = smem_addr(s_tab);
        } else {
            tv.base = tab; tv.saddr = 0;
        }
        const uint32_t *hp = k.head_pack + (size_t)species * HP_TOTAL;
        for (int idx = threadIdx.x; idx < HC_USED; idx += NW * 32) hc[idx] = __uint_as_float(__ldg(hp + HP_TMEM + idx));
        tmem_fill(tm_quarter, hp, warp, lane);
        if (TAB_SMEM) asm volatile("cp.async.wait_group 0;" ::: "memory");
        tmem_fence_before_sync();
        __syncthreads();
        tmem_fence_after_sync();
    };
    // The CTAs start on different central species, in proportion to the species' tiles, so that the species are worked on side by side
    // and most CTAs stage one species only (all CTAs through the species in order / this, one evaluation in us: six equal species, 202,612 atoms
    // 1611 / 1593, 1,000,188 7650 / 7530, 8,001,504 60,470 / 60,010; eight species, tables in global memory, 32,000 atoms 353 / 307,
    // 340,736 2990 / 2999, 2,048,000 17,843 / 17,720).
    // A species whose tiles are all claimed already is passed over: staging its tables would be the only thing left to do.
    volatile int *species_start = ctl + 5;   // [n_species + 1], complete after the staging's barrier
    if ((int)threadIdx.x <= k.n_species) species_start[threadIdx.x] = k.species_dev ? k.species_dev[threadIdx.x] : k.species_start[threadIdx.x];
    // Every group's first tile is fixed (the CTAs that start on a species take its first tiles, group 0 of each before group 1 of any, which
    // spreads a small system over the SMs); the later ones are claimed from the species' counter, which counts from there.
    auto starters = [&](int species) {   // CTAs that start on it
        return k.first_cta[species + 1] - k.first_cta[species];
    };
    int first_species = 0;
    while (first_species + 1 < k.n_species && k.first_cta[first_species + 1] <= (int)blockIdx.x) ++first_species;
    auto species_at = [&](int ss) { return first_species + ss < k.n_species ? first_species + ss : first_species + ss - k.n_species; };
    const int first_tile = (int)blockIdx.x - k.first_cta[first_species] + group * starters(first_species);
    // The first species is staged, and the lists of the first tile's atoms fetched, ahead of the wait for the kernel before this one: they
    // change in list builds only, and the launch after a build does not start early.  864 atoms: 18.8 us from the end of the kernel ahead,
    // 21.7 behind a build, where nothing hides it.
    stage(first_species);
    NextAtoms<APW> nx0;
    int near0 = 0;
    {
        const int s_end0 = species_start[first_species + 1];
        const int slot0 = species_start[first_species] + first_tile * NA + wg + GW * lane;
        nx0.k = &k; nx0.pf = pf; nx0.slot = (lane < APW && slot0 < s_end0) ? slot0 : -1;
        nx0.i = 0; nx0.beg = 0; nx0.len = 0; nx0.use_far = true; nx0.cid = 0;
        nx0.stage_a();
        nx0.template stage_b<L16>();
        if (nx0.slot >= 0) near0 = __ldg(k.nbr_near + nx0.i);
        nx0.template stage_c<L16>(lane);
    }
    wait_previous();
    stamp_begin(k.stamp);
    if (blockIdx.x == 0 && threadIdx.x < (int)(LAUNCH_CLEAR_BYTES / sizeof(double))) k.clear_block[threadIdx.x] = 0.0;
    // lists that an in-step rebuild could not complete (capacity, broken configuration) are not evaluated: the outputs
    // stay at their cleared values and the status word tells the caller why (nothing in this kernel raises these bits,
    // so every CTA takes the same decision)
    const bool skip = (*k.status & (FLAG_NEIGHBOR_OVERFLOW | FLAG_NONFINITE)) != 0;
    const bool use_far = *k.far_flag != 0;   // an atom has moved skin / 4 since the build: every list entry counts
    if (!use_far && nx0.slot >= 0) pf[lane * PF_WORDS + PF_IDX + 3] = near0;   // (the whole lists were fetched: far entries come last)
    __syncwarp();
    for (int ss = 0; ss < k.n_species && !skip; ++ss) {
        const int species = species_at(ss);
        const int s_end = species_start[species + 1];
        if (species_start[species] == s_end) continue;
        auto claimed = [&](int count) { return species_start[species] + (NG * starters(species) + count) * NA; };   // first atom of a claimed tile
        if (ss > 0) {
            // both groups are done with the previous species' tables; the barrier itself carries the decision (a word of shared memory could
            // be written for the next species before a warp has read it: not every turn of this loop has a barrier)
            if (__syncthreads_or(threadIdx.x == 0 && claimed(*reinterpret_cast<volatile int *>(k.tile_counter + species)) >= s_end)) continue;
            stage(species);
        }

        bool prefetched = ss == 0 && __shfl_sync(0xffffffffu, nx0.slot, 0) >= 0;   // this warp's atoms of the coming tile sit in the prefetch buffer
        int look_ahead = -1;       // (group leader) the tile after the current one
        // the group's tiles of this species, each by its first place in the processing order, claimed one ahead: the first is broadcast
        // here, every later one travels with the barrier between encoding and head
        int first = species_start[species] + first_tile * NA;
        if (ss > 0) {
            group_sync(group);
            if (wg == 0 && lane == 0) ctl[2 * group] = claimed(atomicAdd(k.tile_counter + species, 1));
            group_sync(group);
            first = ctl[2 * group];
        }
        while (first < s_end) {
            if (wg == 0 && lane == 0) look_ahead = claimed(atomicAdd(k.tile_counter + species, 1));   // consumed after the encoding
            pc.mark(11);
            const int count = min(NA, s_end - first);

            // ---------------- Encoding + invariants: the warp's atoms wg, wg + 8 ----------------
            if (prefetched) {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                __syncwarp();
            }
            // an atom's moment to tensor memory, its invariants to the regression
            auto finish_atom = [&](int u, const float (&Pf)[4][4]) {
                float *xrow = sX + (wg + GW * u) * X_STRIDE;   // (dE/dG of the last tile's atom: this warp has read it)
                tmem_st16(u == 0 ? tm_p : tm_vt, Pf);
                // Eq. 5 (C_l = I): this lane holds rows a = g, g + 8 of channels 8t + j; sum squares over the rows of a block.
                // Rows 1..3 (l = 1) and 4..7 (l = 2) differ in the top bit of g, so two steps over the lower bits sum both; rows
                // 9..15 (l = 3) take a third.  In each step a lane sends the half of the channels that it does not keep (13 shuffles
                // instead of the 40 of a butterfly: they use the shared-memory pipe).  Row 8 (l = 2), held by g = 0, joins in shared memory.
                const bool g0 = lane & 4, g1 = lane & 8, g2 = lane & 16;
                float qa[8], qb[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float pa = Pf[j & 3][j >> 2], pb = Pf[j & 3][2 + (j >> 2)];
                    qa[j] = g >= 1 ? pa * pa : 0.f;
                    qb[j] = pb * pb;
                }
                if (g == 0) {
                    float4 *to = reinterpret_cast<float4 *>(xrow + 8 * t);
                    to[0] = make_float4(Pf[0][0], Pf[1][0], Pf[2][0], Pf[3][0]);
                    to[1] = make_float4(Pf[0][1], Pf[1][1], Pf[2][1], Pf[3][1]);
                    to[16] = make_float4(qb[0], qb[1], qb[2], qb[3]);
                    to[17] = make_float4(qb[4], qb[5], qb[6], qb[7]);
#pragma unroll
                    for (int j = 0; j < 8; ++j) qb[j] = 0.f;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float sa = g0 ? qa[j] : qa[j + 4], sb = g0 ? qb[j] : qb[j + 4];
                    qa[j] = (g0 ? qa[j + 4] : qa[j]) + __shfl_xor_sync(0xffffffffu, sa, 4);
                    qb[j] = (g0 ? qb[j + 4] : qb[j]) + __shfl_xor_sync(0xffffffffu, sb, 4);
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float sa = g1 ? qa[j] : qa[j + 2], sb = g1 ? qb[j] : qb[j + 2];
                    qa[j] = (g1 ? qa[j + 2] : qa[j]) + __shfl_xor_sync(0xffffffffu, sa, 8);
                    qb[j] = (g1 ? qb[j + 2] : qb[j]) + __shfl_xor_sync(0xffffffffu, sb, 8);
                }
                const float sum3 = (g2 ? qb[1] : qb[0]) + __shfl_xor_sync(0xffffffffu, g2 ? qb[0] : qb[1], 16);
                const int c = 8 * t + (g0 ? 4 : 0) + (g1 ? 2 : 0);   // this lane's channels: c, c + 1; of l = 3 one of them
                xrow[96 + c + (g2 ? 1 : 0)] = sum3;
                __syncwarp();
                float2 *to = reinterpret_cast<float2 *>(xrow + (g2 ? 64 : 32) + c);
                float2 sum = make_float2(qa[0], qa[1]);
                if (g2) { const float2 row8 = *to; sum.x += row8.x; sum.y += row8.y; }
                *to = sum;
                __syncwarp();
                split_invariants(xrow, xs, sc, hc, wg + GW * u, lane);
            };
            const int mine = APW == 1 ? (wg < count) : (wg < count) + (wg + GW < count);   // atoms of this warp
            // Two atoms whose pairs fit the queue together go through the pair loops side by side (see collect_two).
            bool both = false;
            int n0 = 0, n1 = 0, i0 = 0, i1 = 0;
            if (SIDE) {
                if (prefetched && pf[PF_IDX + 3] <= NARROW_CHUNKS * 32 && (mine < 2 || pf[PF_WORDS + PF_IDX + 3] <= NARROW_CHUNKS * 32)) {
                    collect_two<L16>(k, pf, mine, pq, lane, n0, n1);
                    i0 = pf[PF_IDX];
                    i1 = mine == 2 ? pf[PF_WORDS + PF_IDX] : 0;
                    both = true;
                }
            }
            auto atom_and_list = [&](int u, int &i, int64_t &beg, int64_t &end, int &n_pref, int &cs) {
                const int *nidx = pf + u * PF_WORDS;
                n_pref = cs = 0;
                if (prefetched) {
                    i = nidx[PF_IDX];
                    beg = ((int64_t)nidx[PF_IDX + 2] << 32) | (unsigned)nidx[PF_IDX + 1];
                    end = beg + nidx[PF_IDX + 3];
                    n_pref = min(PF_IDX, nidx[PF_IDX + 3]);
                    if (L16) cs = lane < 27 ? nidx[PF_CS + lane] : 0;
                } else {
                    i = (int)MLIP_CHECK_INDEX(__ldg(k.center_order + first + wg + GW * u), k.n, k.status);
                    beg = k.nbr_off[i]; end = use_far ? k.nbr_off[i + 1] : beg + k.nbr_near[i];
                    if (L16) cs = cell_base_of_lane(k, i, lane);
                }
            };
            if (SIDE && !both) {   // longer lists, or the first tile of a species
                both = true;
#pragma unroll 1
                for (int u = 0; u < mine && both; ++u) {
                    int i, n_pref, cs;
                    int64_t beg, end;
                    atom_and_list(u, i, beg, end, n_pref, cs);
                    const double4 pi = load_pos4(k.pos4 + i);
                    const int at = u == 0 ? 0 : (n0 + 15) & ~15;
                    int64_t cur = beg;
                    const int n = collect_pairs<L16>(k, pi, beg, cur, end, pq + at, LY::POOL - at, lane, pf + u * PF_WORDS, n_pref, cs);
                    both = cur >= end;
                    if (u == 0) { n0 = n; i0 = i; } else { n1 = n; i1 = i; }
                }
            }
            if (both) {
                pc.mark(0);
                const int second = (n0 + 15) & ~15, end = second + n1;
                if (lane < 2) *reinterpret_cast<int4 *>(info + 4 * lane) = lane == 0 ? make_int4(i0, n0, 0, 1) : make_int4(i1, n1, second, 1);
                n_pairs += n0 + n1;
                const EncodeLane el(scr, lane);
                int p = 0;   // first pair of the k-step
#pragma unroll 1
                for (int u = 0; u < 2; ++u) {
                    float Pf[4][4];
                    clear_fragments(Pf);
                    const int stop = u == 0 ? n0 : end;
#pragma unroll 1
                    for (; p < stop; p += 16) {
                        if ((p & 16) == 0) {
                            const int slot = p + lane;
                            __syncwarp();
                            encode_rows<TAB_SMEM>(k, tv, pq, slot, slot < n0 || (slot >= second && slot < end), scr, lane);
                            __syncwarp();
                            pc.mark(1);
                        }
                        if (stop - p > 8) encode_kstep<TAB_SMEM, false>(tv, scr, el, (p >> 4) & 1, t, Pf);
                        else encode_kstep<TAB_SMEM, true>(tv, scr, el, (p >> 4) & 1, t, Pf);
                        pc.mark(2);
                    }
                    finish_atom(u, Pf);   // (an empty slot of a ragged tile feeds zeros to the head)
                }
                __syncwarp();
            } else {
                int q_used = 0;   // pairs of the queue that are kept for the derivation
#pragma unroll 1
                for (int u = 0; u < APW; ++u) {
                    float Pf[4][4];
                    if (u < mine) {
                        int i, n_pref, cs, queued = -1;
                        int64_t beg, end;
                        atom_and_list(u, i, beg, end, n_pref, cs);
                        const double4 pi = load_pos4(k.pos4 + i);
                        n_pairs += encode_atom<TAB_SMEM, L16, SIDE ? 1 : 2>(k, tv, pi, beg, end, pq + q_used, LY::POOL - q_used, scr, lane, Pf, queued, pf + u * PF_WORDS, n_pref, cs, pc);
                        if (u + 1 < APW && queued > LY::POOL - SECOND_ROOM) queued = -1;   // leave the next atom room for a scan
                        if (lane == 0) *reinterpret_cast<int4 *>(info + 4 * u) = make_int4(i, queued, q_used, 0);
                        q_used += max(queued, 0);
                    } else {   // empty slot of a ragged tile: feed zeros to the head
                        clear_fragments(Pf);
                        if (u == 0 && lane == 0) *reinterpret_cast<int4 *>(info) = make_int4(0, 0, 0, 0);
                    }
                    finish_atom(u, Pf);
                }
            }
            tmem_wait_st();
            if (wg == 0 && lane == 0) ctl[2 * group + 1] = look_ahead;
            pc.mark(7);
            group_sync(group);
            pc.mark(8);
            const int first_next = ctl[2 * group + 1];

            // ---------------- Regression (and the prefetch for the next tile) ----------------
            NextAtoms<APW> nx;
            nx.k = &k; nx.pf = pf;
            const int next_slot = first_next + wg + GW * lane;
            nx.slot = lane < APW && next_slot < s_end ? next_slot : -1;
            nx.i = 0; nx.beg = 0; nx.len = 0; nx.use_far = use_far; nx.cid = 0;
            head_tile<APW, DET, L16>(k, xs, sX, sc, us, ep, zs, hc, tm_quarter, count, first, group, wg, lane, e_sum, nx, pc);
            prefetched = first_next + wg < s_end;
            pc.mark(9);

            // ---------------- Derivation ----------------
            // W_i = dE_i/dP_i (Eq. 7) of the warp's u-th atom as scaled B fragments; returns the inverse of the scale
            auto weights_of = [&](int u, WFragments &W) {
                const float *drow = sX + (wg + GW * u) * X_STRIDE;   // dE/dG of the atom
                float Pf[4][4];
                tmem_ld16(u == 0 ? tm_p : tm_vt, Pf);
                tmem_wait_ld();
                const int la = g == 0 ? 0 : (g <= 3 ? 1 : 2), lb = g == 0 ? 2 : 3;
                float da[8], db[8];
                {
                    const float4 a0 = *reinterpret_cast<const float4 *>(drow + 32 * la + 8 * t), a1 = *reinterpret_cast<const float4 *>(drow + 32 * la + 8 * t + 4);
                    const float4 b0 = *reinterpret_cast<const float4 *>(drow + 32 * lb + 8 * t), b1 = *reinterpret_cast<const float4 *>(drow + 32 * lb + 8 * t + 4);
                    da[0] = a0.x; da[1] = a0.y; da[2] = a0.z; da[3] = a0.w; da[4] = a1.x; da[5] = a1.y; da[6] = a1.z; da[7] = a1.w;
                    db[0] = b0.x; db[1] = b0.y; db[2] = b0.z; db[3] = b0.w; db[4] = b1.x; db[5] = b1.y; db[6] = b1.z; db[7] = b1.w;
                }
                float w[4][4];   // [nt][0, 1]: row a = g, channels 8t + nt and 8t + 4 + nt; [2, 3]: row g + 8
                float most = 0.f;
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    w[nt][0] = g == 0 ? da[nt] : 2.f * da[nt] * Pf[nt][0];
                    w[nt][1] = g == 0 ? da[4 + nt] : 2.f * da[4 + nt] * Pf[nt][1];
                    w[nt][2] = 2.f * db[nt] * Pf[nt][2];
                    w[nt][3] = 2.f * db[4 + nt] * Pf[nt][3];
                    most = fmaxf(fmaxf(most, fmaxf(fabsf(w[nt][0]), fabsf(w[nt][1]))), fmaxf(fabsf(w[nt][2]), fabsf(w[nt][3])));
                }
                const float sw = scale_for(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(most))));
#pragma unroll
                for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt) {
                        split_h2(w[0][2 * nt + ks] * sw, w[1][2 * nt + ks] * sw, W.hi[ks][nt][0], W.lo[ks][nt][0]);
                        split_h2(w[2][2 * nt + ks] * sw, w[3][2 * nt + ks] * sw, W.hi[ks][nt][1], W.lo[ks][nt][1]);
                    }
                return inverse_pow2(sw);
            };
            auto fold_virial = [&]() {   // deterministic mode: lane sums in a fixed order, then integers
#pragma unroll
                for (int q = 0; q < 9; ++q) {
                    float x = vir[q];
#pragma unroll
                    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                    if (lane == q) vir_fx += rint((double)x * VIRIAL_FX);
                    vir[q] = 0.f;
                }
            };
            const int4 inf0 = *reinterpret_cast<const int4 *>(info);
            if (SIDE && inf0.w != 0) {
                // both atoms' pairs, from the last batch to the first: the second atom's moment, where V and T go, is read before the first of them
                const int4 inf1 = *reinterpret_cast<const int4 *>(info + 4);
                const int second = inf1.z, end = second + inf1.y;
                uint32_t chunk[2];
                derive_chunks(chunk, lane);
                WFragments W;
                float inv0 = 0.f, inv1 = 0.f;
                int holds = -1;   // the atom that W belongs to
                float3 f = make_float3(0.f, 0.f, 0.f);
                bool second_open = inf1.y > 0;
#pragma unroll 1
                for (int p0 = (end - 1) & ~31; p0 >= 0; p0 -= 32) {
                    const int slot = p0 + lane;
                    const bool of_second = slot >= second, live = of_second ? slot < end : slot < inf0.y;
                    derive_rows<TAB_SMEM>(k, tv, pq, slot, live, scr, lane);
                    __syncwarp();
                    pc.mark(4);
#pragma unroll 1
                    for (int mt = p0 + 16 < end ? 1 : 0; mt >= 0; --mt) {
                        const int u = p0 + 16 * mt >= second;
                        if (u != holds) {
                            const float inv = weights_of(u, W);
                            if (u) inv1 = inv; else inv0 = inv;
                            holds = u;
                        }
                        if ((u ? end : inf0.y) - (p0 + 16 * mt) > 8) derive_tile<TAB_SMEM, false>(tv, scr, mt, g, chunk, W, tm_vt);
                        else derive_tile<TAB_SMEM, true>(tv, scr, mt, g, chunk, W, tm_vt);
                    }
                    tmem_wait_st();
                    pc.mark(5);
                    uint32_t vt[32];
                    tmem_ld32(tm_vt, vt);
                    tmem_wait_ld();
                    float3 q = make_float3(0.f, 0.f, 0.f);
                    if (live) q = project_pair<DET>(k, pq[slot], vt, of_second ? inv1 : inv0, vir);
                    if (second_open && p0 <= second) {   // the second atom ends here: what the upper lanes hold is its, the lower ones begin the first's
                        add_own_force<DET>(k, inf1.x, of_second ? make_float3(f.x + q.x, f.y + q.y, f.z + q.z) : f, lane);
                        f = of_second ? make_float3(0.f, 0.f, 0.f) : q;
                        second_open = false;
                    } else {
                        f.x += q.x; f.y += q.y; f.z += q.z;
                    }
                    __syncwarp();
                    pc.mark(6);
                }
                if (inf0.y > 0) add_own_force<DET>(k, inf0.x, f, lane);
                if (DET) fold_virial();
            } else {
                // the second atom first (a rescan of the first one's list would overwrite its queue)
#pragma unroll 1
                for (int u = APW - 1; u >= 0; --u) {
                    if (wg + GW * u >= count) continue;
                    const int4 inf = *reinterpret_cast<const int4 *>(info + 4 * u);
                    WFragments W;
                    const float inv = weights_of(u, W);
                    derive_atom<SIDE, TAB_SMEM, DET, L16>(k, tv, inf.x, pq + inf.z, LY::POOL - inf.z, scr, inf.y, lane, W, inv, vir, tm_vt, pc);
                    if (DET) fold_virial();
                }
            }
            pc.mark(10);
            first = first_next;
        }
    }
    pc.flush(k.acc, lane);

    // totals: per warp into shared memory, per CTA to the global accumulators (from every warp they were 27,000 atomics to one
    // sector of one L2 slice, some 10 us at the end of every launch)
    asm volatile("cp.async.wait_all;" ::: "memory");   // (nothing is left in flight but after a skipped evaluation)
    __syncthreads();   // everybody is done with shared memory
    double *sums = reinterpret_cast<double *>(smem) + warp * TOTALS;   // virial [9], E_i sums of the atoms' lanes, pairs
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        double x = vir_fx;
        if (!DET) {
            float v = vir[q];
#pragma unroll
            for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            x = v;
        }
        if (lane == (DET ? q : 0)) sums[q] = x;
    }
    if (lane < 16) sums[9 + lane] = wg == 7 && lane < NA ? e_sum : 0.0;
    if (lane == 0) reinterpret_cast<unsigned long long *>(sums)[25] = n_pairs;
    tmem_fence_before_sync();
    __syncthreads();
    if (threadIdx.x < TOTALS) {
        const double *col = reinterpret_cast<const double *>(smem) + threadIdx.x;
        if (threadIdx.x == 25) {
            unsigned long long n = 0;
            for (int w = 0; w < NW; ++w) n += reinterpret_cast<const unsigned long long *>(col)[w * TOTALS];
            atomicAdd(k.pair_counter, n);
        } else if (DET) {
            long long x = 0;
            for (int w = 0; w < NW; ++w) x += (long long)col[w * TOTALS];
            atomicAdd(reinterpret_cast<unsigned long long *>(k.acc_fx + (threadIdx.x < 9 ? 1 + threadIdx.x : 0)), (unsigned long long)x);
        } else {
            double x = 0.0;
            for (int w = 0; w < NW; ++w) x += col[w * TOTALS];
            if (x != 0.0) atomicAdd(&k.acc[threadIdx.x < 9 ? ACC_VIRIAL + threadIdx.x : ACC_ENERGY], x);
        }
    }
    stamp_end(k.stamp);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm_base), "r"(TM_COLS) : "memory");
}

// The instantiations, by integer / floating-point scatter and 16-bit / int32 lists; tables in shared memory but for the last.  They are spread over two
// translation units, by measurement: what is compiled beside a kernel decides how its registers are spilled.  With all twelve in one unit (140 bytes
// of spill stores and 172 of loads in the most used kernel, 104 and 116 so), one evaluation in us: one species 432,000 atoms 2795 / 2760, six
// 442,368 3384 / 3341, three 389,344 2483 / 2455, ionic 421,875 2246 / 2220; compact lists 2762 / 2751, 3351 / 3325, 2469 / 2448, 2247 / 2222.  The
// integer scatter of two atoms per warp is the better one beside the kernels of one (19,652 atoms 199 us, on its own 202), the kernels with tables in
// global memory beside those with tables in shared memory (eight species, compact lists, 108,000 atoms 958 us, on their own 978).
using MegaKernel = void (*)(KernelArgs, int);
MegaKernel mega_one(bool det, bool list16);                      // one atom per warp
MegaKernel mega_two_fixed(bool list16);                          // two atoms per warp, side by side; integer scatter
MegaKernel mega_two(bool list16);                                // floating-point scatter
MegaKernel mega_two_global(bool det, bool list16);               // tables in global memory
MegaKernel mega_apart(bool in_smem, bool det, bool list16);      // two atoms per warp, one after the other (launch_megakernel)

}  // namespace mlip
