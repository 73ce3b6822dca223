// Which single traversal builds a system's neighbor lists.  Host arithmetic only: the rule compiles by itself.
#pragma once
#include <stdint.h>

#include <algorithm>

namespace mlip {

// One atom or eight, one after the other, to a warp (tiles of 8 / 64 atoms, k_neighbors_onepass), or one to a lane (tiles of 64, k_neighbors_lanes).
enum class ListForm { WARP_1, WARP_8, LANES };
constexpr int list_form_tile(ListForm f) { return f == ListForm::WARP_1 ? 8 : 64; }

// One atom to a warp in small systems, where eight traversals one after the other are the kernel's time; from there on one to a lane (grids of three
// cells per dimension and more, `rel`).  Whole build on the device in us, one atom to a warp / to a lane: 6 species 6,912 atoms 80 / 126, 10,976 101 /
// 129, 16,384 125 / 128, 32,000 186 / 140; one species 8,192 81 / 113, 16,000 115 / 114, 31,250 164 / 125; three 32,768 176 / 118.
constexpr int64_t LANES_FROM = 18000;
// Where cells hold few atoms a warp's 32 lie in many columns of cells, which its lanes walk one after the other, each a few candidates at a time: not with
// fewer than two atoms to a cell (one where there are tiles enough to hide it), and not where that walk is the kernel's time.  Up to 50,000 atoms one to a warp,
// above that eight / one to a lane: 18,500 atoms of 3 per cell 125 / 141, of 4 119 / 116; 25,000 of 2 155 / 185, of 3 153 / 150; 35,000 of 1 190 / 222, of 2
// 186 / 181; 70,000 of 1 251 / 292, of 2 261 / 242; 100,000 of 1 346 / 377, of 2 358 / 313; 150,000 of 1 462 / 603, of 2 473 / 505 (1.3 rounds of tiles), of 3
// 474 / 394; 300,000 of 1 868 / 944, of 2 877 / 773; 1,000,000 of 1 2807 / 2723, of 1.5 2775 / 2415, of 3 2765 / 1702.
constexpr int64_t LANES_PER_CELL = 2, LANES_SPARSE_FROM = 500000, LANES_WALK = 75000;   // atoms; atoms; atoms times atoms per cell
// Sparse systems and thinner grids, which have no form with an atom to a lane: eight to a warp once such tiles fill the SMs.  Two cells across, one atom to
// a warp / eight: 6 species 19,008 atoms 136 / 194, 26,896 154 / 186, 38,416 195 / 214, 48,400 232 / 303; one species 18,490 114 / 146, 36,000 164 / 165,
// 47,610 208 / 252.  One atom per cell: 50,000 atoms 234 / 223, 70,000 301 / 247, 1,000,000 3712 / 2798.
constexpr int64_t WARP_8_FROM = 50000;

inline ListForm list_form(int64_t n, int64_t n_cells, bool rel) {
    const int64_t per_cell = n < LANES_SPARSE_FROM ? LANES_PER_CELL : 1;
    if (rel && n >= LANES_FROM && n >= per_cell * n_cells && n * n >= LANES_WALK * n_cells) return ListForm::LANES;
    return n < WARP_8_FROM ? ListForm::WARP_1 : ListForm::WARP_8;
}

// Row of a lane (k_neighbors_lanes), in entries, a multiple of four: the mean list at the box's density and 30 percent (lattice shells, composition),
// and where the shared memory of the SMs holds longer rows for all of the tiles at once, those: a list longer than its row is traversed again, and in
// systems of uneven density many are.  Whole build in us with rows from the mean alone / with these: a crystal of 134-entry lists filling half of its box
// 19,652 atoms 252 / 124, 55,296 280 / 150, 78,732 352 / 200; a ball of 26,573 238 / 120; filling its box 19,652 129 / 128, 108,000 271 / 271.
constexpr int LANE_ROW_MOST = 640, LANE_SMEM = 227 * 1024, LANE_SMEM_FIXED = 3 * 1024 + 512;   // per SM; per tile besides the rows (staging, scan, reserved)
inline int list_lane_row(int64_t n, double mean, int sms) {
    const int64_t tiles = (n + 63) / 64, per_sm = (tiles + sms - 1) / sms;
    const int64_t all_at_once = (LANE_SMEM / per_sm - LANE_SMEM_FIXED) / (64 * 2) - 2;
    return (int)std::min(std::max({(int64_t)(1.3 * mean) + 16, all_at_once, (int64_t)64}), (int64_t)LANE_ROW_MOST) / 4 * 4;
}

// Lists whose leading entries (those within r_cut + skin / 2, which evaluations read) are too many for two atoms of a warp to go side by side
// (launch_megakernel): where more than a tenth of them are, or where the density of the box lets the mean list be a tenth longer.
constexpr int LONG_LIST = 96;
inline bool lists_are_long(int64_t n_long, int64_t n_owned) { return 10 * n_long > n_owned; }
inline bool lists_expected_long(double mean) { return mean > 1.1 * LONG_LIST; }

// Look-back words that builds of up to n atoms need, whatever their form.
inline int64_t list_tile_words(int64_t n) { return std::max(n / 64, std::min(n, WARP_8_FROM) / 8) + 2; }

}  // namespace mlip
