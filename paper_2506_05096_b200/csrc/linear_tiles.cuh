// Output tiles of a launch of astraea_gathered_linear (host code only, no CUDA in it).
#pragma once

namespace astraea {

constexpr int kBM = 256;                                 // rows of an output tile: 128 for each CTA of a pair
constexpr int kMaxBN = 256, kBNStep = 32;                // columns of an output tile: what cta_group::2 takes at M = 256

// Columns that a matrix takes in a launch over n_mats of them, and the column tiles of the launch.
inline int mat_columns(int N_out, int n_mats, int bn) { return n_mats == 1 ? 0 : (N_out + bn / 2 - 1) / (bn / 2) * (bn / 2); }
inline int column_tiles(int N_out, int n_mats, int bn) { return ((n_mats == 1 ? N_out : n_mats * mat_columns(N_out, n_mats, bn)) + bn - 1) / bn; }

// Columns of an output tile.  The launch takes ceil(tiles / pairs) rounds, and a round of narrower tiles costs less, but
// not in proportion (the rows of x are streamed for fewer columns): measured 0.60-0.67 of a 256-column round at 128
// columns on seven shapes.  256 unless another width saves 3 % by that estimate, which happens where a launch has a
// few rounds only or the last tile of a row is mostly padding.  Several matrices: half a tile is whole groups of 32 columns, since
// the epilogue's groups must not straddle two matrices.
inline int choose_bn(long long rows, int N_out, int n_mats, int pairs)
{
    const long long tiles_m = (rows + kBM - 1) / kBM;
    int best_bn = kMaxBN;
    double best = 0.0;
    for (int bn = kMaxBN; bn >= kBNStep; bn -= n_mats == 1 ? kBNStep : 64) {
        const long long tiles = tiles_m * column_tiles(N_out, n_mats, bn);
        const double t = (double)((tiles + pairs - 1) / pairs) * (0.26 + 0.74 * bn / kMaxBN);
        if (best == 0.0 || t < 0.97 * best) { best = t; best_bn = bn; }
    }
    return best_bn;
}

}  // namespace astraea
