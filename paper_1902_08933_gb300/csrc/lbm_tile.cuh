// lbm_tile.cuh -- the fused step on small two-dimensional tiles, for domains too
// small to fill the GPU with row marches.
//
// A row march (lbm_device.cuh, lbm_step_x2.cuh) forms the rows of its run one
// after the other, each behind two block barriers: with the 8 rows a run that
// keep its halo cheap, a step of a 64 x 64 grid is a serial chain of about 12
// rows on 8 of the 152 SMs. Here a block owns a tile of at most 128 cells (FP64,
// odd nx: one cell a thread) or 128 pairs of cells (FP32 arithmetic, nx even) and
// takes every row at once, in three phases with a barrier between them:
//   A. every load of the tile is issued together: its own h, g, phi u and p (kept
//      in registers until the collision) and the h of the 2-cell halo ring; phi
//      of the tile and its halo into shared memory, p with a 1-cell halo;
//   B. mu (Eq. 8) of the tile and a 1-cell ring;
//   C. the collision and push of the tile's cells.
// The halo costs 1.7 to 3 loads of h a cell, from L2 where the grid fits there; FP64
// runs larger grids on tiles too, bound by its operations either way. The arithmetic is that of the marches, cell by cell (phi in the same
// order of summation, chem_pot, macroscopic, collide_emit).
//
// One cooperative launch runs several steps: block b takes items b, b + gridDim,
// ... of every step, and before step s > 0 of an item waits (bounded, as in
// step_kernel_x2_multi) until the items within 3 cells of it have finished step
// s - 1: one step reads h up to 2 cells outside the tile, which cells up to 3
// outside have pushed, and pushes 1 cell out, into what cells up to 3 outside
// read. Items of one step never wait on one another and every block is resident,
// so every wait ends.
#pragma once

#include "lbm_device.cuh"
#include "lbm_step_x2.cuh"

namespace lbm {

constexpr int kTileThreads = 128;

// Shared memory of a tile of up to 2^ulog units (cells or pairs) a row, all its
// rows: rows of RW entries, column x at x - x0 + 4 (pairs on 8-byte boundaries).
template <typename R, int CPT, bool COMP>
struct TileSmem {
    // the largest of (columns + 8) x (rows + 4) over the shapes 2^u units x 128 / 2^u rows
    static constexpr int entries = CPT == 1 ? 40 * 8 > 12 * 36 ? 40 * 8 : 12 * 36 : 72 * 8 > 16 * 36 ? 72 * 8 : 16 * 36;
    R phi[entries], mu[entries], p[entries];
    R lo[COMP ? entries : 1];
};

// Position of halo unit k of a tile of `rows` rows and nu units of CPT columns
// (nu + 4 / CPT units a row with the halo): rows above and below first, then the
// side columns. ry, rx: row and first column relative to the tile.
template <int CPT>
struct TileHalo {
    int w, rows, np, nsu;   // columns; rows; units of a full halo row; side units a row
    __device__ __forceinline__ TileHalo(int w_, int rows_)
        : w(w_), rows(rows_), np((w_ + 4) / CPT), nsu(4 / CPT) {}
    // ring of `depth` rows (2: phi; 1: mu): number of units and unit k's position
    __device__ __forceinline__ int count(int depth) const { return 2 * depth * np + rows * nsu; }
    __device__ __forceinline__ void at(int depth, int k, int& ry, int& rx) const {
        const int caps = 2 * depth * np;
        if (k < caps) {
            const int q = k / np;
            ry = q < depth ? q - depth : rows + q - depth;
            rx = (k - q * np) * CPT - 2;
        } else {
            k -= caps;
            ry = k / nsu;
            const int side = k - ry * nsu;
            rx = side < nsu / 2 ? side * CPT - 2 : w + (side - nsu / 2) * CPT;
        }
    }
};

// ---------------------------------------------------------------------------
// Two cells a thread: the FP32-arithmetic forms, nx even.
template <int FORM>
__device__ __forceinline__ void tile_item_x2(const StepArgs& a, const Consts<float>& C, const WorkItem& wk, int ulog,
                                             TileSmem<float, 2, Form<FORM>::comp>& sm, int tid, bool swap) {
    using F = Form<FORM>;
    using HT = typename F::HT;
    using GT = typename F::GT;
    const int U = 1 << ulog, RW = 2 * U + 8;
    const int nx = C.nx, ny = C.ny, walls = C.walls, base = (int)C.base;
    const int x0 = wk.x0, y0 = wk.ystart, w = wk.dir, rows = wk.nrows;
    const long long S = a.S;
    const long long sw = swap ? a.set_delta : 0;
    auto moved = [sw](const void* p, long long sign) {
        return static_cast<const void*>(static_cast<const char*>(p) + sign * sw);
    };
    const HT* hin = static_cast<const HT*>(moved(a.h_in, 1));
    const float2* h0in = static_cast<const float2*>(moved(a.h0_in, 1));
    const GT* gin = static_cast<const GT*>(moved(a.g_in, 1));
    const float* p_in = static_cast<const float*>(moved(a.p_in, 1));
    float* phiu = static_cast<float*>(a.phiu);
    const X2Out<FORM> out{static_cast<HT*>(const_cast<void*>(moved(a.h_out, -1))),
                          static_cast<float2*>(const_cast<void*>(moved(a.h0_out, -1))),
                          static_cast<GT*>(const_cast<void*>(moved(a.g_out, -1))), phiu,
                          static_cast<float*>(const_cast<void*>(moved(a.p_out, -1))), S};
    auto wrapx = [nx](int x) { return x < 0 ? x + nx : (x >= nx ? x - nx : x); };
    // the stored row of row y: mirrored at walls (reading Q7), wrapped otherwise
    auto rowg = [ny, walls](int y) {
        if (walls) return y < 0 ? -1 - y : (y >= ny ? 2 * ny - 1 - y : y);
        return y < 0 ? y + ny : (y >= ny ? y - ny : y);
    };
    const TileHalo<2> H(w, rows);
    const int tx = tid & (U - 1), ty = tid >> ulog;
    const bool act = 2 * tx < w && ty < rows;
    const int X = x0 + 2 * tx, Y = y0 + ty;
    const int c = act ? base + Y * nx + X : 0;

    // phi of the pair at cell offset cc (hv: its h as stored; lo: low parts), Eq. 18
    auto phi_at = [&](int cc, F2 (&hv)[9], F2& lo) {
        if constexpr (F::cons) {
            const float4 h0 = *reinterpret_cast<const float4*>(h0in + cc);
#pragma unroll
            for (int i = 1; i < 9; ++i) hv[i] = ld_pair(hin + (long long)(i - 1) * S + cc);
            F2 s8 = F2(0.f);
#pragma unroll
            for (int i = 1; i < 9; ++i) s8 = s8 + hv[i];
            if constexpr (F::h16) s8 = s8 * C.ihs;   // exact: a power of two
            float sa, ea, ha, la, sb, eb, hb, lb;
            two_sum(h0.x, s8.v.x, sa, ea);
            fast_two_sum(sa, ea + h0.y, ha, la);
            two_sum(h0.z, s8.v.y, sb, eb);
            fast_two_sum(sb, eb + h0.w, hb, lb);
            lo = F2(la, lb);
            hv[0] = lo;
            return F2(ha, hb);
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) hv[i] = ld_pair(hin + (long long)i * S + cc);
            F2 phi = hv[0];
#pragma unroll
            for (int i = 1; i < 9; ++i) phi = phi + hv[i];
            return phi;
        }
    };
    auto put = [&](int ry, int rx, F2 phi, F2 lo, F2 p) {
        const int j = (ry + 2) * RW + rx + 4;
        st_pair(sm.phi + j, phi);
        st_pair(sm.p + j, p);
        if constexpr (F::comp) st_pair(sm.lo + j, lo);
    };
    // A. the thread's own pair, then its share of the halo ring (threads without
    // a pair of their own first)
    F2 h[9], g[9], pux = F2(0.f), puy = F2(0.f), lo = F2(0.f);
    if (act) {
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = ld_pair(gin + (long long)i * S + c);
        pux = ld_pair(phiu + c);
        puy = ld_pair(phiu + S + c);
        const F2 p = ld_pair(p_in + c);
        const F2 phi = phi_at(c, h, lo);
        put(ty, 2 * tx, phi, lo, p);
    }
    const int own = U * rows;
    const int h0 = tid >= own ? tid - own : tid + kTileThreads - own;
    for (int k = h0; k < H.count(2); k += kTileThreads) {
        int ry, rx;
        H.at(2, k, ry, rx);
        const int cc = base + rowg(y0 + ry) * nx + wrapx(x0 + rx);
        F2 hv[9], l = F2(0.f);
        const F2 p = ld_pair(p_in + cc);
        const F2 phi = phi_at(cc, hv, l);
        put(ry, rx, phi, l, p);
    }
    __syncthreads();
    // B. mu; a ghost row's is its mirror row's
    auto mu_at = [&](int ry, int rx) {
        const int y = y0 + ry;
        const int cr = walls ? rowg(y) - y0 : ry;
        const int j = (cr + 2) * RW + rx + 4;
        Nbr<F2> n;
        nbr_pair(sm.phi - RW, sm.phi, sm.phi + RW, j, n);
        F2 mu;
        if constexpr (F::comp) {
            Nbr<F2> nl;
            nbr_pair(sm.lo - RW, sm.lo, sm.lo + RW, j, nl);
            mu = chem_pot2(C, n.z[1][1], nl.z[1][1], n.lap() + nl.lap());
        } else {
            mu = chem_pot(C, n.z[1][1], n.lap());
        }
        st_pair(sm.mu + (ry + 2) * RW + rx + 4, mu);
    };
    if (act) mu_at(ty, 2 * tx);
    for (int k = h0; k < H.count(1); k += kTileThreads) {
        int ry, rx;
        H.at(1, k, ry, rx);
        mu_at(ry, rx);
    }
    __syncthreads();
    // C. collision and push
    if (!act) return;
    const int j = (ty + 2) * RW + 2 * tx + 4;
    auto rowoff = [&](int y) { return base + rowg(y) * nx; };
    auto load_nbr = [&](Nbr<F2>& nphi, Nbr<F2>& nmu, Nbr<F2>& np) {
        nbr_pair(sm.phi - RW, sm.phi, sm.phi + RW, j, nphi);
        nbr_pair(sm.mu - RW, sm.mu, sm.mu + RW, j, nmu);
        nbr_pair(sm.p - RW, sm.p, sm.p + RW, j, np);
    };
    auto load_h = [&](F2 (&hv)[9], F2& l) {
#pragma unroll
        for (int i = 0; i < 9; ++i) hv[i] = h[i];
        l = lo;
    };
    MonAcc<F2> mon;
    x2_collide_push<FORM, 0>(C, out, Y, X, wrapx(X - 1), wrapx(X + 2), rowoff, load_nbr, load_h, g, pux, puy, mon);
}

// ---------------------------------------------------------------------------
// One cell a thread: FP64, and the FP32-arithmetic forms with nx odd.
template <int FORM>
__device__ __forceinline__ void tile_item_1(const StepArgs& a, const Consts<typename Form<FORM>::R>& C,
                                            const WorkItem& wk, int ulog,
                                            TileSmem<typename Form<FORM>::R, 1, false>& sm, int tid, bool swap) {
    using F = Form<FORM>;
    using R = typename F::R;
    using AT = typename F::AT;
    const int U = 1 << ulog, RW = U + 8;
    const int nx = C.nx, ny = C.ny, walls = C.walls, base = (int)C.base;
    const int x0 = wk.x0, y0 = wk.ystart, w = wk.dir, rows = wk.nrows;
    const long long sw = swap ? a.set_delta : 0;
    auto moved = [sw](const void* p, long long sign) {
        return static_cast<const void*>(static_cast<const char*>(p) + sign * sw);
    };
    PopIO<F> io;
    io.hin = static_cast<const typename F::HT*>(moved(a.h_in, 1));
    io.hout = static_cast<typename F::HT*>(const_cast<void*>(moved(a.h_out, -1)));
    io.h0in = static_cast<const float2*>(moved(a.h0_in, 1));
    io.h0out = static_cast<float2*>(const_cast<void*>(moved(a.h0_out, -1)));
    io.gin = static_cast<const typename F::GT*>(moved(a.g_in, 1));
    io.gout = static_cast<typename F::GT*>(const_cast<void*>(moved(a.g_out, -1)));
    io.S = a.S; io.hs = C.hs; io.ihs = C.ihs; io.gs = C.gs; io.igs = C.igs;
    const AT* p_in = static_cast<const AT*>(moved(a.p_in, 1));
    AT* p_out = static_cast<AT*>(const_cast<void*>(moved(a.p_out, -1)));
    AT* phiu = static_cast<AT*>(a.phiu);
    auto wrapx = [nx](int x) { return x < 0 ? x + nx : (x >= nx ? x - nx : x); };
    auto rowg = [ny, walls](int y) {
        if (walls) return y < 0 ? -1 - y : (y >= ny ? 2 * ny - 1 - y : y);
        return y < 0 ? y + ny : (y >= ny ? y - ny : y);
    };
    const TileHalo<1> H(w, rows);
    const int tx = tid & (U - 1), ty = tid >> ulog;
    const bool act = tx < w && ty < rows;
    const int X = x0 + tx, Y = y0 + ty;
    const int c = act ? base + Y * nx + X : 0;
    R h[9], g[9], pux = R(0), puy = R(0);
    if (act) {
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = io.load_g(i, c);
        pux = R(phiu[c]);
        puy = R(phiu[a.S + c]);
        const int j = (ty + 2) * RW + tx + 4;
        sm.p[j] = R(p_in[c]);
        R lo;
        sm.phi[j] = io.phi_of(c, h, lo);
        if constexpr (F::cons) h[0] = lo;   // low part of phi
    }
    const int own = U * rows;
    const int h0 = tid >= own ? tid - own : tid + kTileThreads - own;
    for (int k = h0; k < H.count(2); k += kTileThreads) {
        int ry, rx;
        H.at(2, k, ry, rx);
        const int cc = base + rowg(y0 + ry) * nx + wrapx(x0 + rx);
        const int j = (ry + 2) * RW + rx + 4;
        R hv[9], lo;
        sm.p[j] = R(p_in[cc]);
        sm.phi[j] = io.phi_of(cc, hv, lo);
    }
    __syncthreads();
    auto nbr = [&](const R* f, int j, Nbr<R>& n) {
#pragma unroll
        for (int dy = 0; dy < 3; ++dy)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) n.z[dy][dx] = f[j + (dy - 1) * RW + dx - 1];
    };
    auto mu_at = [&](int ry, int rx) {
        const int cr = walls ? rowg(y0 + ry) - y0 : ry;   // a ghost row's mu is its mirror row's
        Nbr<R> n;
        nbr(sm.phi, (cr + 2) * RW + rx + 4, n);
        if constexpr (sizeof(R) == 8) sm.mu[(ry + 2) * RW + rx + 4] = chem_pot_f64(C, n);
        else sm.mu[(ry + 2) * RW + rx + 4] = chem_pot(C, n.z[1][1], n.lap());
    };
    if (act) mu_at(ty, tx);
    for (int k = h0; k < H.count(1); k += kTileThreads) {
        int ry, rx;
        H.at(1, k, ry, rx);
        if (rx >= -1 && rx <= w) mu_at(ry, rx);
    }
    __syncthreads();
    if (!act) return;
    const int j = (ty + 2) * RW + tx + 4;
    Nbr<R> nphi, nmu, np;
    nbr(sm.phi, j, nphi);
    nbr(sm.mu, j, nmu);
    nbr(sm.p, j, np);
    const bool bot = walls && Y == 0, top = walls && Y == ny - 1;
    MonAcc<R> mon;
    collide_push<F, false>(C, io, phiu, p_out, base + Y * nx, bot ? 0 : base + rowg(Y - 1) * nx,
                           top ? 0 : base + rowg(Y + 1) * nx, bot, top, X, wrapx(X - 1), wrapx(X + 1), nphi, nmu, np, h,
                           g, pux, puy, mon);
}

// Several steps of a tile plan. OCC: the resident blocks a SM the registers are
// sized for; the planner (plan_tile) takes, for pairs, 3 (168 registers: more of
// a tile's loads in flight) while every item then has a block of its own, else 4
// (128 registers, no spills). Measured, LBM_F32_C, us a step: 64 x 64 3.8 with 3
// and 4.2 with 4; 512 x 512 (1024 items) 15.7 with 3, 12.9 with 4, 18.5 with 5.
// FP64 runs 2 (255 registers): 512 x 512 121 us against 130 with 3, 139 with 4.
template <int FORM, bool PAIR, int OCC>
__global__ void __launch_bounds__(kTileThreads, OCC) step_kernel_tile(const StepArgs a) {
    using R = typename Form<FORM>::R;
    __shared__ __align__(16) TileSmem<R, PAIR ? 2 : 1, PAIR && Form<FORM>::comp> sm;
    __shared__ int s_bad;
    const int tid = threadIdx.x;
    int* abort_flag = a.done + a.ndesc;
    Consts<R> C;
    int inst = -1;
    for (int s = 0; s < a.nsteps; ++s) {
        for (int item = blockIdx.x; item < a.ndesc; item += gridDim.x) {
            const WorkItem wk = a.work[item];
            if (wk.inst != inst) {
                inst = wk.inst;
                C.load(a.inst[inst]);
            }
            if (s > 0 && !tile_wait(a.done, a.nbr + item * kMaxTileNbr, s + a.wait_extra, a.wait_limit, a.status,
                                    abort_flag, &s_bad, tid))
                return;
            if constexpr (PAIR) tile_item_x2<FORM>(a, C, wk, a.tile_ulog, sm, tid, (s & 1) != 0);
            else tile_item_1<FORM>(a, C, wk, a.tile_ulog, sm, tid, (s & 1) != 0);
            __syncthreads();   // every thread's stores of the step issued, the rings free
            if (tid == 0 && a.nsteps > 1) {
                __threadfence();
                atomicExch(a.done + item, s + 1);
            }
        }
    }
}

}  // namespace lbm
