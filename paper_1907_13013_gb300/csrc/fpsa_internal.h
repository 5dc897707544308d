// Internal declarations shared by the library's host driver and kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/fpsa.h"

namespace fpsa {

// S_N tables (host, FP64). Matrices row-major N x N; moments padded to N.
struct Tables {
    int N = 0, L1 = 0;
    std::vector<double> mu, w;
    std::vector<double> D;    // D[l][n] = w_n P_l(mu_n)
    std::vector<double> M;    // M[n][l] = (2l+1)/2 P_l(mu_n), zero for l >= L1
    std::vector<double> Afp;  // discrete angular Laplacian (MPD or WFD)
};
void build_tables(int N, int L1, int laplacian, Tables &t);

// Columns per block of the few-column tensor-core contractions (tc_contract.cuh): the fewest
// (of 16, 32, 64) whose blocks fit one per SM; 0: the 128-column tiles. A wider block costs
// more the more outputs a thread holds, whatever the order, while the tiles' time falls with
// it, most below N = 65, where they hold both operators and all inputs of a tile at once. Us
// for the pair of kernels of an iteration, few-column form against tiles, one right-hand side:
//   N =          16           32           48           64           96           128
//   CT = 16      11.6 / 11.7  11.6 / 15.2               13.1 / 22.8               14.5 / 88
//   CT = 32      15.8 / 11.7  15.6 / 15.1  17.3 / 19.2  17.0 / 22.9               19.3 / 96
//   CT = 64      30.6 / 12.1  51.9 / 15.9               55.0 / 23.1  56.3 / 81.8  57.3 / 96
inline int col_tile(int N, int sumK, int R, int n_sm) {
    const int widest = N <= 32 ? 16 : (N <= 64 ? 32 : 64);
    for (int ct = 16; ct <= widest; ct *= 2)
        if (((2ll * sumK + ct - 1) / ct) * R <= n_sm) return ct;
    return 0;
}

// Whether the GMRES vector kernels take small chunks (kDotChunkSmall elements a block) instead
// of large ones (kDotChunk): where the small ones are few. A block's fixed work, the meeting
// of its threads' sums for every four vectors, is paid per chunk, and in FP32 a small chunk is
// one 16-byte word a thread. Vector kernels of 40 Krylov steps (FP32, two restarts) and 20
// (FP64), us, large / small chunks, by the number of small blocks:
//   FP32  125: 3407 / 2960   300: 3472 / 3443   600: 3727 / 4686   1125: 4051 / 7091
//   FP64  125: 4069 / 1740   300: 4174 / 2108   600: 4439 / 3099    900: 4922 / 4099   1125: 5093 / 5234
inline bool small_dot_chunks(long long small_blocks, bool fp64, int n_sm) { return small_blocks <= (fp64 ? 6ll : 2ll) * n_sm; }

// One cell eliminated at one block-cyclic-reduction level (or an instance root).
// Cell ids are global (concatenated over instances); -1 = absent.
// Coupling slots index the per-level N/2 x N/2 coupling blocks B (to the left
// neighbour's right-node mu>0 values) and C (to the right neighbour's left-node
// mu<0 values): slot(j, l) = slot_base[j] + l.
struct BcrItem {
    int32_t cell, left, right;
    int32_t s_cell;        // slot(cell, l)
    int32_t s_left;        // slot(left, l)
    int32_t s_left_next;   // slot(left, l+1)
    int32_t s_right;       // slot(right, l)
    int32_t s_right_next;  // slot(right, l+1)
    int32_t local;         // cell index within its instance
    int32_t K_inst;        // cells of the instance
    int32_t level;         // level the cell is eliminated at (roots: the instance's level count)
};

// Device-side geometry of the batch.
struct Geometry {
    int B = 0, N = 0, L1 = 0, R = 0, sumK = 0, Kmax = 0;
    int n_levels = 0;                   // max over instances
    int n_slots = 0;
    std::vector<int32_t> K, off;        // per instance
    std::vector<int32_t> cell_inst;     // per global cell
    std::vector<int32_t> slot_base;     // per global cell
    std::vector<std::vector<BcrItem>> levels;  // [level] -> items over all instances
    std::vector<BcrItem> roots;         // one per instance
};
void build_geometry(const int32_t *K, int B, int N, int L1, int R, Geometry &g);

}  // namespace fpsa
