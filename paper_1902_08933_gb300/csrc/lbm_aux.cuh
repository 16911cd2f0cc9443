// lbm_aux.cuh -- the kernels around the time step: the initial state, the
// macroscopic fields for read-back, the FP64 diagnostics and the population
// dump. Off the hot loop; they reuse the cell arithmetic of lbm_device.cuh.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

// ---------------------------------------------------------------------------
// Initial state (reading Q6): h = h^eq(phi0, mu0, u = 0), g = g^eq(p = 0, u = 0)
// (all zero with rho_0 = 0), phi*u of the previous step 0, p 0.
template <int FORM>
__global__ void init_kernel(const StepArgs a, const double* __restrict__ phi0, int instance) {
    using F = Form<FORM>;
    using R = typename F::R;
    using AT = typename F::AT;
    Consts<R> C;
    C.load(a.inst[instance]);
    PopIO<F> io;
    io.hout = static_cast<typename F::HT*>(a.h_out);
    io.h0out = static_cast<float2*>(a.h0_out);
    io.gout = static_cast<typename F::GT*>(a.g_out);
    io.S = a.S; io.hs = C.hs; io.ihs = C.ihs; io.gs = C.gs; io.igs = C.igs;
    AT* phiu = static_cast<AT*>(a.phiu);
    AT* p0 = static_cast<AT*>(a.p_out);
    AT* p1 = static_cast<AT*>(const_cast<void*>(a.p_in));
    const int n = C.nx * C.ny;
    for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < n; cell += gridDim.x * blockDim.x) {
        const int x = cell % C.nx, y = cell / C.nx;
        Nbr<R> nb;
        for (int dy = -1; dy <= 1; ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                int yy = y + dy, xx = x + dx;
                xx = xx < 0 ? xx + C.nx : (xx >= C.nx ? xx - C.nx : xx);
                if (C.walls) yy = yy < 0 ? -1 - yy : (yy >= C.ny ? 2 * C.ny - 1 - yy : yy);
                else yy = yy < 0 ? yy + C.ny : (yy >= C.ny ? yy - C.ny : yy);
                nb.z[dy + 1][dx + 1] = R(phi0[yy * C.nx + xx]);
            }
        const R phi = nb.z[1][1];
        const R mu = chem_pot(C, phi, nb.lap());
        const R etamu = C.eta * mu;
        const long long c = C.base + cell;
        R hv[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) hv[i] = (i == 0) ? phi + (w_of<R>(0) - R(1)) * etamu : w_of<R>(i) * etamu;
        if constexpr (F::cons) {
            // h_0 = phi_0 - sum of the stored h_1..8, exactly as a float pair
            double rest = 0.0;
#pragma unroll
            for (int i = 1; i < 9; ++i) { hv[i] = io.round_h(hv[i]); rest += double(hv[i]); }
            const double h0 = phi0[cell] - rest;
            const float hi = float(h0);
            io.store_h0(c, make_float2(hi, float(h0 - double(hi))));
        } else {
            io.store_h(0, c, hv[0]);
        }
#pragma unroll
        for (int i = 1; i < 9; ++i) io.store_h(i, c, hv[i]);
#pragma unroll
        for (int i = 0; i < 9; ++i) io.store_g(i, c, R(0));
        phiu[c] = AT(0);
        phiu[a.S + c] = AT(0);
        p0[c] = AT(0);
        p1[c] = AT(0);
    }
}

// ---------------------------------------------------------------------------
// Macroscopic fields and diagnostics of one instance, in three passes over
// global memory (phi, then mu, then everything else; the fields of small domains
// in one, fields_tile) -- off the hot loop. They
// compute in FP64 whatever the storage form: the stored populations convert to
// FP64 exactly (phi of the conservative forms from its two-float h_0 to about
// 2^-48), so the fields, sums and the Laplace pressure P of Sec. 4.2 measure the
// stored state without adding FP32 rounding of their own.
template <int FORM>
__global__ void phi_pass(const AuxArgs a) {
    using F = Form<FORM>;
    using R = typename F::R;
    Consts<R> C;
    C.load(a.inst[a.instance]);
    PopIO<F> io;
    io.hin = static_cast<const typename F::HT*>(a.h);
    io.h0in = static_cast<const float2*>(a.h0);
    io.S = a.S; io.hs = C.hs; io.ihs = C.ihs;
    const int n = C.nx * C.ny;
    for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < n; cell += gridDim.x * blockDim.x) {
        const long long c = C.base + cell;
        R hv[9], lo;
        const R phi = io.phi_of(c, hv, lo);
        a.tmp_phi[cell] = double(phi) + double(lo);
    }
}

// 3x3 neighbourhood of a field (x periodic; y periodic or mirrored at walls)
template <typename T>
__device__ __forceinline__ void gather(const T* f, int nx, int ny, int walls, int x, int y, Nbr<double>& nb) {
    const int xs[3] = {x == 0 ? nx - 1 : x - 1, x, x == nx - 1 ? 0 : x + 1};
    const int ys[3] = {y == 0 ? (walls ? 0 : ny - 1) : y - 1, y, y == ny - 1 ? (walls ? ny - 1 : 0) : y + 1};
#pragma unroll
    for (int dy = 0; dy < 3; ++dy)
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) nb.z[dy][dx] = double(f[ys[dy] * nx + xs[dx]]);
}

template <int FORM>
__global__ void mu_pass(const AuxArgs a) {
    Consts<double> C;
    C.load(a.inst[a.instance]);
    const int n = C.nx * C.ny;
    for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < n; cell += gridDim.x * blockDim.x) {
        Nbr<double> nb;
        gather(a.tmp_phi, C.nx, C.ny, C.walls, cell % C.nx, cell / C.nx, nb);
        a.tmp_mu[cell] = chem_pot_f64(C, nb);
    }
}

// Everything one cell's macroscopic stage produces, plus (PLAP) the Laplace-law P
// of Sec. 4.2. FIN: also whether every population is finite. Bound by its FP64
// operations (macroscopic_f64), like the FP64 step: what is not asked for is not
// formed.
template <int FORM, bool PLAP, bool FIN>
__device__ __forceinline__ void cell_fields(const AuxArgs& a, const Consts<double>& C, int x, int y,
                                            const Nbr<double>& nphi, const Nbr<double>& nmu, double out[7],
                                            bool& finite) {
    using F = Form<FORM>;
    using SR = typename F::R;   // the storage form's arithmetic type: the values as loaded
    using AT = typename F::AT;
    PopIO<F> io;
    io.hin = static_cast<const typename F::HT*>(a.h);
    io.h0in = static_cast<const float2*>(a.h0);
    io.gin = static_cast<const typename F::GT*>(a.g);
    io.S = a.S; io.hs = SR(C.hs); io.ihs = SR(C.ihs); io.gs = SR(C.gs); io.igs = SR(C.igs);
    const long long c = C.base + y * C.nx + x;
    Nbr<double> np;
    gather(static_cast<const AT*>(a.p_prev) + C.base, C.nx, C.ny, C.walls, x, y, np);
    double g[9];
    finite = true;
    g[0] = 0.0;
#pragma unroll
    for (int i = FIN ? 0 : 1; i < 9; ++i) {   // g_0 enters no field
        g[i] = double(io.load_g(i, c));       // exact: FP16 or FP32 times a power of two
        if constexpr (FIN) finite = finite && isfinite(g[i]);
    }
    if constexpr (FIN) {
        SR hv[9], lo;
        io.phi_of(c, hv, lo);
        finite = finite && isfinite(lo);
#pragma unroll
        for (int i = 0; i < 9; ++i) finite = finite && isfinite(hv[i]);
    }
    const MacroD m = macroscopic_f64(C, g, nphi, nmu, np);
    const double phi = nphi.z[1][1];
    out[0] = phi; out[1] = m.ux.v; out[2] = m.uy.v; out[3] = m.p.v; out[4] = m.rho.v; out[5] = nmu.z[1][1];
    out[6] = 0.0;
    if constexpr (PLAP) {
        // P = p_0 - kappa phi lap(phi) + kappa |grad phi|^2 / 2 + p, p_0 = phi psi' - psi (Sec. 4.2)
        const double psi = C.beta * phi * phi * (phi - 1.0) * (phi - 1.0);
        const double dpsi = 2.0 * C.beta * phi * (phi - 1.0) * (2.0 * phi - 1.0);
        out[6] = (phi * dpsi - psi) - C.kappa6 * phi * lap6(nphi).v +
                 (0.5 / 144.0) * C.kappa * fmadd(m.Gx, m.Gx, m.Gy * m.Gy).v + m.p.v;
    }
}

// The same with phi and mu from the scratch planes.
template <int FORM, bool PLAP, bool FIN>
__device__ __forceinline__ void cell_fields_at(const AuxArgs& a, const Consts<double>& C, int cell, double out[7],
                                               bool& finite) {
    const int x = cell % C.nx, y = cell / C.nx;
    Nbr<double> nphi, nmu;
    gather(a.tmp_phi, C.nx, C.ny, C.walls, x, y, nphi);
    gather(a.tmp_mu, C.nx, C.ny, C.walls, x, y, nmu);
    cell_fields<FORM, PLAP, FIN>(a, C, x, y, nphi, nmu, out, finite);
}

__device__ __forceinline__ void put_fields(const AuxArgs& a, int n, int cell, const double v[7]) {
    int k = 0;
    for (int b = 0; b < 7; ++b)
        if (a.mask & (1u << b)) a.out[(long long)(k++) * n + cell] = v[b];
}

template <int FORM, bool PLAP>
__global__ void fields_pass(const AuxArgs a) {
    Consts<double> C;
    C.load(a.inst[a.instance]);
    const int n = C.nx * C.ny;
    for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < n; cell += gridDim.x * blockDim.x) {
        double v[7];
        bool fin;
        cell_fields_at<FORM, PLAP, false>(a, C, cell, v, fin);
        put_fields(a, n, cell, v);
    }
}

// The three passes in one launch, a block a tile of kFieldTX x kFieldTY cells: phi of
// the tile and a halo of 2 cells and mu of a halo of 1 in shared memory, mirrored at
// walls as gather() does. Three launches are most of the time of a small domain
// (64 x 64 20.6 -> 10.4 us, 150 x 150 20.6 -> 16.5); a large one is bound by its FP64
// operations, of which the halo adds 0.4 of the mu of a cell, and takes the passes
// (launch_fields_t). 16 x 8 cells: enough blocks at the sizes this serves.
constexpr int kFieldTX = 16, kFieldTY = 8;
template <int FORM, bool PLAP>
__global__ void __launch_bounds__(kFieldTX * kFieldTY) fields_tile(const AuxArgs a) {
    using F = Form<FORM>;
    using R = typename F::R;
    constexpr int PW = kFieldTX + 4, MW = kFieldTX + 2;
    __shared__ double s_phi[(kFieldTY + 4) * PW], s_mu[(kFieldTY + 2) * MW];
    Consts<double> C;
    C.load(a.inst[a.instance]);
    const int nx = C.nx, ny = C.ny, walls = C.walls;
    const int strips = (nx + kFieldTX - 1) / kFieldTX;
    const int x0 = (int)blockIdx.x % strips * kFieldTX, y0 = (int)blockIdx.x / strips * kFieldTY;
    const int w = min(kFieldTX, nx - x0), rows = min(kFieldTY, ny - y0);
    auto wrapx = [nx](int x) { return x < 0 ? x + nx : (x >= nx ? x - nx : x); };
    auto rowg = [ny, walls](int y) {
        if (walls) return y < 0 ? -1 - y : (y >= ny ? 2 * ny - 1 - y : y);
        return y < 0 ? y + ny : (y >= ny ? y - ny : y);
    };
    auto nbr = [](const double* f, int j, int width, Nbr<double>& n) {
#pragma unroll
        for (int dy = 0; dy < 3; ++dy)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) n.z[dy][dx] = f[j + (dy - 1) * width + dx - 1];
    };
    PopIO<F> io;
    io.hin = static_cast<const typename F::HT*>(a.h);
    io.h0in = static_cast<const float2*>(a.h0);
    io.S = a.S; io.hs = R(C.hs); io.ihs = R(C.ihs);
    for (int k = threadIdx.x; k < (rows + 4) * PW; k += kFieldTX * kFieldTY) {
        const int ry = k / PW - 2, rx = k % PW - 2;
        if (rx >= w + 2) continue;
        R hv[9], lo;
        const R phi = io.phi_of(C.base + rowg(y0 + ry) * nx + wrapx(x0 + rx), hv, lo);
        s_phi[k] = double(phi) + double(lo);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < (rows + 2) * MW; k += kFieldTX * kFieldTY) {
        const int ry = k / MW - 1, rx = k % MW - 1;
        if (rx > w) continue;
        const int cr = walls ? rowg(y0 + ry) - y0 : ry;   // a ghost row's mu is its mirror row's
        Nbr<double> nb;
        nbr(s_phi, (cr + 2) * PW + rx + 2, PW, nb);
        s_mu[k] = chem_pot_f64(C, nb);
    }
    __syncthreads();
    const int tx = threadIdx.x % kFieldTX, ty = threadIdx.x / kFieldTX;
    if (tx >= w || ty >= rows) return;
    Nbr<double> nphi, nmu;
    nbr(s_phi, (ty + 2) * PW + tx + 2, PW, nphi);
    nbr(s_mu, (ty + 1) * MW + tx + 1, MW, nmu);
    double v[7];
    bool fin;
    cell_fields<FORM, PLAP, false>(a, C, x0 + tx, y0 + ty, nphi, nmu, v, fin);
    put_fields(a, nx * ny, (y0 + ty) * nx + x0 + tx, v);
}

// Diagnostics: per-block FP64 partial sums written to a.partials (scratch,
// kDiagBlocks x kDiagQuantities), then one block adds the partials in a fixed
// order, so the result does not depend on timing.
//   0 sum phi, 1 sum rho, 2 kinetic energy, 3 max |u|, 4 sum phi x, 5 sum phi y,
//   6 sum (1-phi) x, 7 sum (1-phi) y, 8 sum P (bulk A), 9 n bulk A,
//   10 sum P (bulk B), 11 n bulk B, 12 non-finite count, 13 sum (1 - phi)
__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}

template <int FORM>
__global__ void __launch_bounds__(256) diag_pass(const AuxArgs a) {
    Consts<double> C;
    C.load(a.inst[a.instance]);
    const int n = C.nx * C.ny;
    double acc[kDiagQuantities];
#pragma unroll
    for (int q = 0; q < kDiagQuantities; ++q) acc[q] = 0.0;
    for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < n; cell += gridDim.x * blockDim.x) {
        double v[7];
        bool fin;
        cell_fields_at<FORM, true, true>(a, C, cell, v, fin);
        const double phi = v[0], ux = v[1], uy = v[2], rho = v[4], P = v[6];
        const double x = double(cell % C.nx), y = double(cell / C.nx);
        const double uu = ux * ux + uy * uy;
        acc[0] += phi;
        acc[1] += rho;
        acc[2] += 0.5 * rho * uu;
        acc[3] = fmax(acc[3], sqrt(uu));
        acc[4] += phi * x;
        acc[5] += phi * y;
        acc[6] += (1.0 - phi) * x;
        acc[7] += (1.0 - phi) * y;
        if (phi > 1.0 - 1e-3) { acc[8] += P; acc[9] += 1.0; }
        if (phi < 1e-3) { acc[10] += P; acc[11] += 1.0; }
        if (!fin) acc[12] += 1.0;
        acc[13] += 1.0 - phi;
    }
    __shared__ double red[kDiagQuantities][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < kDiagQuantities; ++q) {
        const double v = (q == 3) ? warp_max(acc[q]) : warp_sum(acc[q]);
        if (lane == 0) red[q][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < kDiagQuantities) {
        const int q = threadIdx.x;
        double v = red[q][0];
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) v = (q == 3) ? fmax(v, red[q][k]) : v + red[q][k];
        a.partials[blockIdx.x * kDiagQuantities + q] = v;
    }
}

// Final sum of the per-block partials: thread t takes blocks t, t + 256, ...,
// then a fixed shuffle / shared-memory tree combines the threads.
constexpr int kDiagFinalThreads = 256;
static __global__ void __launch_bounds__(kDiagFinalThreads) diag_final(const double* __restrict__ partials,
                                                                       int nblocks, double* __restrict__ result) {
    const int t = threadIdx.x;
    double acc[kDiagQuantities];
#pragma unroll
    for (int q = 0; q < kDiagQuantities; ++q) acc[q] = 0.0;
    for (int b = t; b < nblocks; b += kDiagFinalThreads)
#pragma unroll
        for (int q = 0; q < kDiagQuantities; ++q) {
            const double x = partials[b * kDiagQuantities + q];
            acc[q] = (q == 3) ? fmax(acc[q], x) : acc[q] + x;
        }
    __shared__ double red[kDiagQuantities][kDiagFinalThreads / 32];
    const int lane = t & 31, warp = t >> 5;
#pragma unroll
    for (int q = 0; q < kDiagQuantities; ++q) {
        const double v = (q == 3) ? warp_max(acc[q]) : warp_sum(acc[q]);
        if (lane == 0) red[q][warp] = v;
    }
    __syncthreads();
    if (t < kDiagQuantities) {
        double v = red[t][0];
        for (int w = 1; w < kDiagFinalThreads / 32; ++w) v = (t == 3) ? fmax(v, red[t][w]) : v + red[t][w];
        result[t] = v;
    }
}

template <int FORM>
__global__ void populations_pass(const AuxArgs a, double* out_h, double* out_g) {
    using F = Form<FORM>;
    using R = typename F::R;
    Consts<R> C;
    C.load(a.inst[a.instance]);
    PopIO<F> io;
    io.hin = static_cast<const typename F::HT*>(a.h);
    io.h0in = static_cast<const float2*>(a.h0);
    io.gin = static_cast<const typename F::GT*>(a.g);
    io.S = a.S; io.hs = C.hs; io.ihs = C.ihs; io.gs = C.gs; io.igs = C.igs;
    const int n = C.nx * C.ny;
    for (int cell = blockIdx.x * blockDim.x + threadIdx.x; cell < n; cell += gridDim.x * blockDim.x) {
        const long long c = C.base + cell;
        for (int i = 0; i < 9; ++i) {
            if (out_h) {
                double v;
                if (F::cons && i == 0) {
                    const float2 h0 = io.load_h0(c);
                    v = double(h0.x) + double(h0.y);
                } else {
                    v = double(io.load_h(i, c));
                }
                out_h[(long long)i * n + cell] = v;
            }
            if (out_g) out_g[(long long)i * n + cell] = double(io.load_g(i, c));
        }
    }
}

}  // namespace lbm
