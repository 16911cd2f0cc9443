// lbm_tileplan.h -- host side of the plans that run several steps a launch: domains
// cut into tiles (step_kernel_tile, sp_tile_kernel), and the neighbours of each tile
// and of each item of a row march (step_kernel_x2_multi).
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

// What a launch of several steps keeps on the device: its items (those of a row march
// are the context's, nwork = 0), their neighbours, and the steps finished per item
// followed by the abort flag. One allocation or none.
struct ItemBuffers {
    void* base = nullptr;
    WorkItem* work = nullptr;
    int *nbr = nullptr, *done = nullptr;
    // alloc(void**, bytes): whether it was had
    template <typename Alloc>
    bool allocate(size_t nwork, size_t items, Alloc&& alloc) {
        auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
        const size_t wb = up(nwork * sizeof(WorkItem)), nb = up(items * kMaxTileNbr * sizeof(int));
        void* p = nullptr;
        *this = ItemBuffers();
        if (!alloc(&p, wb + nb + (items + 1) * sizeof(int)) || !p) return false;
        base = p;
        work = reinterpret_cast<WorkItem*>(p);
        nbr = reinterpret_cast<int*>(static_cast<char*>(p) + wb);
        done = reinterpret_cast<int*>(static_cast<char*>(p) + wb + nb);
        return true;
    }
    void release() {
        cudaFree(base);
        *this = ItemBuffers();
    }
    // Allocates and fills them. cudaErrorMemoryAllocation (cleared): there is no room,
    // and the plan that wanted them is not made.
    cudaError_t upload(const std::vector<WorkItem>& items, const std::vector<int>& neighbours) {
        release();
        const size_t n = neighbours.size() / kMaxTileNbr;
        cudaError_t e = cudaSuccess;
        if (!allocate(items.size(), n, [&e](void** p, size_t b) { return (e = cudaMalloc(p, b)) == cudaSuccess; })) {
            cudaGetLastError();
            return e;
        }
        if (!items.empty()) e = cudaMemcpy(work, items.data(), items.size() * sizeof(WorkItem), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(nbr, neighbours.data(), neighbours.size() * sizeof(int), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemset(done, 0, (n + 1) * sizeof(int));
        if (e != cudaSuccess) release();
        return e;
    }
};

struct Domain {
    int nx, ny;
    bool per_y;   // periodic in y (in x always)
};

// Neighbours of the items of a row march, strips of tx columns (dom(instance): its
// Domain): for each item the other items of its instance within the 3 cells that a
// step reaches -- it reads h up to 2 cells outside the item, which cells up to 3
// outside have pushed --, kMaxTileNbr an item, -1 padded. A last strip may be as
// narrow as 2 columns, so the item beyond it counts too. False: one has more.
template <typename Dom>
bool march_neighbours(const WorkItem* items, int count, int tx, Dom&& dom, std::vector<int>& nbr) {
    struct Box { int inst, x0, x1, y0, y1; };
    std::vector<Box> box(count);
    for (int k = 0; k < count; ++k) {
        const WorkItem& w = items[k];
        const int y0 = w.dir < 0 ? w.ystart - w.nrows + 1 : w.ystart;
        box[k] = {w.inst, w.x0, std::min(dom(w.inst).nx, w.x0 + tx), y0, y0 + w.nrows};
    }
    // [a0, a1) and [b0, b1) meet, with b shifted by -n, 0, +n when periodic
    auto meet = [](int a0, int a1, int b0, int b1, int n, bool periodic) {
        for (int sh = periodic ? -1 : 0; sh <= (periodic ? 1 : 0); ++sh)
            if (b0 + sh * n < a1 && a0 < b1 + sh * n) return true;
        return false;
    };
    nbr.assign((size_t)count * kMaxTileNbr, -1);
    for (int k = 0; k < count; ++k) {
        const Domain d = dom(box[k].inst);
        int cnt = 0;
        for (int m = 0; m < count; ++m) {
            if (m == k || box[m].inst != box[k].inst) continue;
            if (!meet(box[k].x0 - 3, box[k].x1 + 3, box[m].x0, box[m].x1, d.nx, true)) continue;
            if (!meet(box[k].y0 - 3, box[k].y1 + 3, box[m].y0, box[m].y1, d.ny, d.per_y)) continue;
            if (cnt == kMaxTileNbr) return false;
            nbr[(size_t)k * kMaxTileNbr + cnt++] = m;
        }
    }
    return true;
}

// Steps of one launch: 256 at most, and what the batched queue can count -- steps x
// items, past which every block counts on once, stay below 2^31.
constexpr int kLaunchSteps = 256;
inline int batched_steps(int left, int items) {
    constexpr int kMost = 0x7fffffff - (1 << 20);   // (1 << 20: more blocks than are ever resident)
    return std::max(1, std::min(std::min(left, kLaunchSteps), kMost / std::max(1, items)));
}

// Calls f(rows) for each run length that cuts ny rows into equal runs, the longest
// (one run) first, until it returns false: the different values of ceil(ny / r),
// about 2 sqrt(ny) of them.
template <typename F>
void each_run_length(int ny, F&& f) {
    for (long long r = 1; r <= ny;) {
        const int rows = (int)((ny + r - 1) / r);
        if (!f(rows) || rows == 1) return;
        r = (ny + (long long)rows - 2) / (rows - 1);   // the first r of a shorter run
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
