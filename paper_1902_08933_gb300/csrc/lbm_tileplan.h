// lbm_tileplan.h -- host side of the tile plans (step_kernel_tile, sp_tile_kernel):
// domains cut into tiles and each tile's neighbours.
#pragma once

#include <algorithm>
#include <vector>

#include "lbm_internal.h"

namespace lbm {

struct TileList {
    std::vector<WorkItem> items;   // dir: columns of the tile
    std::vector<int> nbr;          // kMaxTileNbr an item, -1 padded
};

// Tiles of a domain: its columns (in units of cpt cells) cut into equal parts of
// at most U units, its rows into equal parts of at most R -- parts of at least 2
// cells, so that the tiles within the 3 cells a step reaches (x periodic, y where
// per_y) are at most two away.
inline void add_tiles(TileList& out, int inst, int nx, int ny, int cpt, bool per_y, int U, int R) {
    const int nu = nx / cpt, kx = (nu + U - 1) / U, ky = (ny + R - 1) / R;
    auto xcut = [&](int i) { return (int)((long long)nu * i / kx) * cpt; };   // part i: [cut(i), cut(i + 1))
    auto ycut = [&](int i) { return (int)((long long)ny * i / ky); };
    // parts within 3 cells of part i along one axis (itself among them)
    auto near_parts = [](int m, int n, bool periodic, auto&& cut) {
        std::vector<std::vector<int>> v(m);
        for (int i = 0; i < m; ++i)
            for (int j = i - 2; j <= i + 2; ++j) {
                if (!periodic && (j < 0 || j >= m)) continue;
                const int q = ((j % m) + m) % m, sh = (j - q) / m * n;   // part q, moved by whole periods
                if (cut(q) + sh >= cut(i + 1) + 3 || cut(i) - 3 >= cut(q + 1) + sh) continue;
                if (std::find(v[i].begin(), v[i].end(), q) == v[i].end()) v[i].push_back(q);
            }
        return v;
    };
    const auto nearx = near_parts(kx, nx, true, xcut);
    const auto neary = near_parts(ky, ny, per_y, ycut);
    const int first = (int)out.items.size();
    for (int j = 0; j < ky; ++j)
        for (int i = 0; i < kx; ++i) {
            WorkItem w;
            w.inst = inst;
            w.x0 = xcut(i);
            w.dir = xcut(i + 1) - w.x0;
            w.ystart = ycut(j);
            w.nrows = ycut(j + 1) - w.ystart;
            w.pad = 0;
            out.items.push_back(w);
            const size_t at = out.nbr.size();
            for (int jj : neary[j])
                for (int ii : nearx[i])
                    if (ii != i || jj != j) out.nbr.push_back(first + jj * kx + ii);
            out.nbr.resize(at + kMaxTileNbr, -1);   // at most 5 x 5 - 1
        }
}

// The smallest of 8 x 4, 8 x 8 and 16 x 8 units whose tiles (count(U, R) of them)
// leave no SM with two; else 16 x 8.
template <typename Count>
inline void tile_shape(Count&& count, int sms, int* U, int* R) {
    *U = 16;
    *R = 8;
    const int shapes[3][2] = {{8, 4}, {8, 8}, {16, 8}};
    for (const auto& s : shapes)
        if (count(s[0], s[1]) <= sms) {
            *U = s[0];
            *R = s[1];
            return;
        }
}

}  // namespace lbm
