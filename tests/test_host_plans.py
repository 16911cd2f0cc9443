"""Host code of the plans, compiled by itself and run on the CPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1902_08933_gb300", "csrc")


def run_cpp(tmp_path, code):
    """Compiles code (C++, the headers of csrc/) and runs it; its output."""
    from paper_1902_08933_gb300 import build
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(code)
    r = subprocess.run([cxx, "-std=c++17", "-O2", "-Wall", "-Werror", "-I", CSRC, "-isystem", cuda, str(src), "-o",
                        str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    return r.stdout


def test_persistent_monitor_buffers_come_all_or_not_at_all(tmp_path):
    run_cpp(tmp_path, r"""
#include <cstdint>
#include <cstdlib>
#include "lbm_monbuf.h"
using lbm::kMonQ;
using lbm::kMonSub;
int main() {
    for (size_t steps : {1, 64}) for (size_t items : {1, 7, 456}) for (size_t n : {1, 3}) {
        lbm::MultiMonitor m;
        int calls = 0;
        if (m.allocate(steps, items, n, [&](void**, size_t) { ++calls; return false; })) return 1;
        if (calls != 1 || m.slots || m.sub || m.count) return 2;
        size_t bytes = 0;
        void* base = nullptr;
        if (!m.allocate(steps, items, n, [&](void** p, size_t b) { bytes = b; base = *p = std::malloc(b); return true; })) return 3;
        const char *b0 = (char*)base, *s = (char*)m.slots, *u = (char*)m.sub, *c = (char*)m.count;
        const size_t ns = steps * items * kMonQ * 8, nu = steps * n * kMonSub * kMonQ * 8, nc = steps * n * (kMonSub + 1) * 4;
        if (s != b0 || u < s + ns || c < u + nu || c + nc > b0 + bytes) return 4;
        if ((uintptr_t)u % 8 || (uintptr_t)c % 4) return 5;
        // a second attempt that fails leaves nothing of the first
        std::free(base);
        if (m.allocate(steps, items, n, [](void**, size_t) { return false; }) || m.slots || m.sub || m.count) return 6;
    }
    return 0;
}
""")


NEIGHBOURS = r"""
#include <cstdio>
#include <set>
#include "lbm_tileplan.h"
using lbm::WorkItem;
// The items' neighbour lists against every pair of cells within 3 of one another.
struct Rect { int x0, x1, y0, y1; };
static int check(const std::vector<Rect>& r, const std::vector<int>& nbr, int nx, int ny, bool per_y) {
    std::vector<int> owner((size_t)nx * ny, -1);
    for (int k = 0; k < (int)r.size(); ++k)
        for (int y = r[k].y0; y < r[k].y1; ++y)
            for (int x = r[k].x0; x < r[k].x1; ++x) {
                if (owner[y * nx + x] >= 0) return 1;
                owner[y * nx + x] = k;
            }
    std::vector<std::set<int>> want(r.size());
    for (int y = 0; y < ny; ++y)
        for (int x = 0; x < nx; ++x) {
            if (owner[y * nx + x] < 0) return 2;
            for (int dy = -3; dy <= 3; ++dy)
                for (int dx = -3; dx <= 3; ++dx) {
                    int Y = y + dy;
                    if (!per_y && (Y < 0 || Y >= ny)) continue;
                    Y = (Y + 2 * ny) % ny;
                    want[owner[y * nx + x]].insert(owner[Y * nx + (x + dx + 2 * nx) % nx]);
                }
        }
    for (int k = 0; k < (int)r.size(); ++k) {
        std::set<int> got;
        for (int j = 0; j < lbm::kMaxTileNbr; ++j)
            if (nbr[(size_t)k * lbm::kMaxTileNbr + j] >= 0) got.insert(nbr[(size_t)k * lbm::kMaxTileNbr + j]);
        want[k].erase(k);
        if (got != want[k]) {
            std::printf("%d x %d periodic %d: item %d has %zu neighbours for %zu\n", nx, ny, per_y, k, got.size(), want[k].size());
            return 3;
        }
    }
    return 0;
}
"""


def test_march_neighbours_are_the_items_within_three_cells(tmp_path):
    # a last strip of 1 to 4 columns beside whole ones, one strip, runs of few rows
    run_cpp(tmp_path, NEIGHBOURS + r"""
int main() {
    for (int tx : {64, 128, 256})
        for (int nx : {tx, tx + 2, tx + 4, 2 * tx + 2, 3 * tx + 2, 2 * tx, tx / 2, 6, 3})
            for (int rows : {8, 9, 5, 3})
                for (int ny : {3, 8, 16, 17, 40})
                    for (bool per_y : {false, true}) {
                        std::vector<WorkItem> w;
                        std::vector<Rect> r;
                        for (int x0 = 0; x0 < nx; x0 += tx)
                            for (int y0 = 0, k = 0; y0 < ny; y0 += rows, ++k) {
                                const int y1 = std::min(ny, y0 + rows);
                                WorkItem i{};
                                i.x0 = x0;
                                i.nrows = y1 - y0;
                                i.dir = k % 2 ? 1 : -1;
                                i.ystart = i.dir < 0 ? y1 - 1 : y0;
                                w.push_back(i);
                                r.push_back({x0, std::min(nx, x0 + tx), y0, y1});
                            }
                        std::vector<int> nbr;
                        if (!lbm::march_neighbours(w.data(), (int)w.size(), tx, [&](int) { return lbm::Domain{nx, ny, per_y}; }, nbr))
                            return 9;
                        if (int e = check(r, nbr, nx, ny, per_y)) return e;
                    }
    return 0;
}
""")


def test_tile_neighbours_are_the_tiles_within_three_cells(tmp_path):
    run_cpp(tmp_path, NEIGHBOURS + r"""
int main() {
    const int shapes[4][2] = {{8, 4}, {8, 8}, {16, 8}, {8, 16}};
    for (auto& s : shapes)
        for (int cpt : {1, 2})
            for (int nx = 3; nx < 75; nx += nx < 40 ? 1 : 7)
                for (int ny : {3, 4, 5, 7, 8, 9, 15, 16, 17, 18, 33, 34, 50})
                    for (bool per_y : {false, true}) {
                        if (nx % cpt) continue;
                        lbm::TileList list;
                        lbm::add_tiles(list, 0, nx, ny, cpt, per_y, s[0], s[1]);
                        std::vector<Rect> r;
                        for (const WorkItem& w : list.items) {
                            if (w.dir > s[0] * cpt || w.nrows > s[1]) return 9;
                            r.push_back({w.x0, w.x0 + w.dir, w.ystart, w.ystart + w.nrows});
                        }
                        if (int e = check(r, list.nbr, nx, ny, per_y)) return e;
                    }
    return 0;
}
""")


def test_run_lengths_are_those_of_every_number_of_runs(tmp_path):
    # the different ceil(ny / r) in order; the tallest grids accepted take few calls
    run_cpp(tmp_path, r"""
#include "lbm_tileplan.h"
int main() {
    for (int ny = 1; ny < 2000; ++ny) {
        std::vector<int> want, got;
        for (int r = 1; r <= ny; ++r)
            if (want.empty() || want.back() != (ny + r - 1) / r) want.push_back((ny + r - 1) / r);
        lbm::each_run_length(ny, [&](int rows) { got.push_back(rows); return true; });
        if (got != want) return 1;
    }
    for (int ny : {79536431, 715827882, 2147483647}) {
        long long calls = 0;
        int last = 0;
        lbm::each_run_length(ny, [&](int rows) { ++calls; last = rows; return true; });
        if (last != 1 || calls > 100000) return 2;
        calls = 0;
        lbm::each_run_length(ny, [&](int rows) { ++calls; return rows >= 8; });
        if (calls > 100000) return 3;
    }
    return 0;
}
""")


def test_item_buffers_come_all_or_not_at_all(tmp_path):
    run_cpp(tmp_path, r"""
#include <cstdint>
#include <cstdlib>
#include "lbm_tileplan.h"
extern "C" cudaError_t cudaFree(void*) { return cudaSuccess; }
int main() {
    for (size_t nwork : {0, 1, 11, 456}) for (size_t items : {1, 11, 456}) {
        lbm::ItemBuffers b;
        if (b.allocate(nwork, items, [](void**, size_t) { return false; }) || b.base || b.work || b.nbr || b.done) return 1;
        size_t bytes = 0;
        if (!b.allocate(nwork, items, [&](void** p, size_t n) { *p = std::malloc(bytes = n); return true; })) return 2;
        const char *w = (char*)b.work, *n = (char*)b.nbr, *d = (char*)b.done;
        if (w != b.base || n < w + nwork * sizeof(lbm::WorkItem) || d < n + items * lbm::kMaxTileNbr * sizeof(int)) return 3;
        if (d + (items + 1) * sizeof(int) > w + bytes || (uintptr_t)n % 4 || (uintptr_t)d % 4) return 4;
        std::free(b.base);
        b.release();
        if (b.base || b.work || b.nbr || b.done) return 5;
    }
    return 0;
}
""")


def test_batched_queue_counts_stay_below_2_31(tmp_path):
    # 1.1e9 cells in items of 128 x 1 (run length 1 asked for) are 8.6 million items a step
    run_cpp(tmp_path, r"""
#include "lbm_tileplan.h"
int main() {
    for (long long items : {1LL, 700LL, 8000000LL, 8388608LL, 8600000LL, 16777216LL, 2000000000LL})
        for (int left : {1, 2, 255, 256, 257, 100000}) {
            const int n = lbm::batched_steps(left, (int)items);
            if (n < 1 || n > left || n > 256) return 1;
            if (n * items + (1 << 20) > 0x7fffffffLL) return 2;
            if (items < 8000000 && n != (left < 256 ? left : 256)) return 3;
        }
    return 0;
}
""")
