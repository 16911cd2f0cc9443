// lbm_sp.cu -- the single-phase models of Sec. 2.3 on the D2Q9 lattice: the
// generalized lattice Boltzmann model with a mass source, in the forms of
// Remarks 3, 1 and 2, and the explicit D_i G_i scheme of Remark 4.
//
// Remark 3 (model LBM_SP_INCOMPRESSIBLE_SOURCE): rho~ = rho_0 and a constant
// density (rho = 1), the incompressible Navier-Stokes equations with a mass
// source (div u = S) and a uniform body force: the cell's populations and source
// give u (Eq. 27a) and p (Eq. 28 with G_0), the equilibrium (Eq. 25 with rho~ =
// rho_0, rho = 1; g_0 stored shifted by rho_0) and the force term
//   G_i = w_i { S + c_i.F / c_s^2 + (c_i c_i - c_s^2 I):(u F + F u + Q S I) / (2 c_s^4) },
//   Q = (2/d) c_s^2 - xi / (tau_g - 1/2),
// then BGK (Eq. 24) and push-streaming (x periodic; y periodic or halfway
// bounce-back walls). Storage and arithmetic in FP64 or FP32.
//
// Remark 1 (LBM_SP_NEARLY_INCOMPRESSIBLE; rho~ = rho, p = rho c_s^2): rho =
// sum g + S/2 (Eq. 27aa), u = (sum c g + F/2) / rho, g^eq = rho (w_i + s_i(u))
// (Eq. 29bb), G_i with (u F + F u - u u S + Q div(u) I) and Q = (2/d) rho c_s^2 -
// xi / (tau_g - 1/2); div u by Eq. 30a (mirror at walls). The populations are
// stored as g_i - w_i (their rest state at rho = 1), so that FP32 storage keeps
// the small deviations that carry the flow: rho = 1 + sum(g - w) + S/2.
//
// Remark 2 (LBM_SP_HE_INCOMPRESSIBLE): the same with g in units of pressure (g^eq
// = w_i p + p_0 s_i(u), Eq. 29bd; p_0 S_1 and p_0 F_1), stored as g_i - w_i p_0.
//
// Remark 4 (scheme LBM_SP_SCHEME_REMARK4): the Remark 3 model with a
// velocity-dependent force F(u) = F_0 - (lambda + beta |u|) u, evolved with the
// explicit D_i G_i (unshifted f, u = sum c f). G_i at the destination x + c_i is
// the destination's own, which its thread forms from its f; G_i(x, t - 1) is
// formed again from u at t - 1 (two planes kept instead of the nine planes of G).
//
// Every step is one kernel: Remark 3 one unit a thread, the others a row march or,
// in small domains, tiles for several steps. A unit is a cell, or in FP32 with nx
// even two horizontally adjacent cells in packed FP32 instructions. The cell
// arithmetic (sp_moments_of, sp_collide) is written once for all of them.
#include <cmath>
#include <cstring>
#include <string>

#include "lbm.h"
#include "lbm_mbar.cuh"
#include "lbm_tileplan.h"
#include "lbm_device.cuh"   // lbm::F2, two cells' FP32 values in packed instructions

namespace {

using lbm::F2;
constexpr int kQ = 9;
__host__ __device__ constexpr int sx(int i) { return i == 1 || i == 5 || i == 8 ? 1 : (i == 3 || i == 6 || i == 7 ? -1 : 0); }
__host__ __device__ constexpr int sy(int i) { return i == 2 || i == 5 || i == 6 ? 1 : (i == 4 || i == 7 || i == 8 ? -1 : 0); }
__host__ __device__ constexpr double sw(int i) { return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0); }
__host__ __device__ constexpr int sopp(int i) { return i == 0 ? 0 : (i <= 4 ? (i + 1) % 4 + 1 : (i - 5 + 2) % 4 + 5); }
static_assert(sopp(1) == 3 && sopp(2) == 4 && sopp(5) == 7 && sopp(6) == 8 && sopp(8) == 6, "D2Q9 opposites");
// one direction of each opposite pair (1, 2, 5, 6; their opposites 3, 4, 7, 8)
__host__ __device__ constexpr int pair2(int q) { return q == 0 ? 1 : q == 1 ? 2 : q == 2 ? 5 : 6; }

struct SpConst {
    int nx, ny, walls;
    double inv_tau, src, tgm, Qc, fx, fy;   // 1/tau_g, 1 - 1/(2 tau_g), tau_g - 1/2, Q, F
    double dl, dq;                          // drag of the Remark 4 scheme: F(u) = F - (dl + dq |u|) u
    double p0;                              // Remark 2: the constant p_0
    // derived on the host, so that FP32 kernels do no FP64 arithmetic on them
    double tau, Qd0;                        // tau_g; Q - (2/d) c_s^2 (the part of Q without the density)
    double hp0, ip0, hp0fx, hp0fy;          // p_0 / 2, 1 / p_0, p_0 F_1 / 2
};

template <typename R>
struct SpCell { R ux, uy, p; };

// u (Eq. 27a, rho = 1), G_i (Remark 3) and p (Eq. 28) of one cell
template <typename R>
__device__ __forceinline__ SpCell<R> sp_moments(const SpConst& K, const R g[kQ], R S, R G[kQ]) {
    SpCell<R> m;
    R jx = R(0), jy = R(0), rest = R(0);
#pragma unroll
    for (int i = 1; i < kQ; ++i) {
        if (sx(i)) jx += sx(i) > 0 ? g[i] : -g[i];
        if (sy(i)) jy += sy(i) > 0 ? g[i] : -g[i];
        rest += g[i];
    }
    const R fx = R(K.fx), fy = R(K.fy);
    m.ux = jx + R(0.5) * fx;
    m.uy = jy + R(0.5) * fy;
    const R uF = m.ux * fx + m.uy * fy, uu = m.ux * m.ux + m.uy * m.uy;
    const R QS = R(K.Qc) * S;
    // (c c - c_s^2 I):(u F + F u + Q S I) / (2 c_s^4) = 9 (c.u)(c.F) - 3 u.F + 4.5 (|c|^2 - 2/3) Q S;
    // for opposite directions the part even in c is shared and c.F / c_s^2 flips sign
    G[0] = R(sw(0)) * (S - R(3) * uF + R(4.5) * (-R(2.0 / 3.0)) * QS);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = pair2(q), j = sopp(i);
        const R cu = R(sx(i)) * m.ux + R(sy(i)) * m.uy, cF = R(sx(i)) * fx + R(sy(i)) * fy;
        const R c2 = R(sx(i) * sx(i) + sy(i) * sy(i));
        const R e = R(sw(i)) * (S + R(9) * cu * cF - R(3) * uF + R(4.5) * (c2 - R(2.0 / 3.0)) * QS);
        const R o = R(sw(i)) * (R(3) * cF);
        G[i] = e + o;
        G[j] = e - o;
    }
    // Eq. 28: c_s^2 / (1 - w_0) = 3/5; s_0(u) = -w_0 u.u / (2 c_s^2) = -(2/3) u.u
    m.p = R(0.6) * (rest + R(0.5) * S - R(2.0 / 3.0) * uu + R(K.tgm) * G[0]);
    return m;
}

// ---- Remarks 1 and 2 (M = 1, 2) ----
// g holds g_i - w_i a0 (a0 = 1 for Remark 1, p_0 for Remark 2: the rest state).
// d = rho - 1 (Remark 1) or p - p_0 (Remark 2); a = rho or p_0, the factor of
// s_i(u) in g^eq (Eq. 29bb, Eq. 29bd); both equilibria are d w_i + a s_i(u)
// after the shift. Sg and the force Fg are in the units of g (Remark 2: p_0 S_1,
// p_0 F_1).
template <int M, typename R>
__device__ __forceinline__ void sp1_moments(const SpConst& K, const R g[kQ], R S, R& d, R& a, R& ux, R& uy) {
    R m0 = g[0], jx = R(0), jy = R(0);
#pragma unroll
    for (int i = 1; i < kQ; ++i) {
        m0 += g[i];
        if (sx(i)) jx += sx(i) > 0 ? g[i] : -g[i];
        if (sy(i)) jy += sy(i) > 0 ? g[i] : -g[i];
    }
    if constexpr (M == 1) {
        d = m0 + R(0.5) * S;                       // Eq. 27aa
        a = R(1) + d;
        const R ir = R(1) / a;
        ux = (jx + R(0.5) * R(K.fx)) * ir;         // Eq. 27a
        uy = (jy + R(0.5) * R(K.fy)) * ir;
    } else {
        d = m0 + R(K.hp0) * S;                     // p = sum g + p_0 S_1 / 2
        a = R(K.p0);
        ux = (jx + R(K.hp0fx)) * R(K.ip0);         // p_0 u = sum c g + p_0 F_1 / 2
        uy = (jy + R(K.hp0fy)) * R(K.ip0);
    }
}

template <int M, typename R>
__global__ void sp1_fields_kernel(const R* __restrict__ g, const R* __restrict__ src, long long N, SpConst K,
                                  unsigned mask, double* __restrict__ out) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    R gc[kQ], d, a, ux, uy;
#pragma unroll
    for (int i = 0; i < kQ; ++i) gc[i] = g[i * N + c];
    sp1_moments<M>(K, gc, src[c], d, a, ux, uy);
    // Remark 1: p = rho c_s^2, rho = 1 + d; Remark 2: p = p_0 + d
    const double p = M == 1 ? (1.0 + double(d)) / 3.0 : K.p0 + double(d);
    int slot = 0;
    if (mask & LBM_FIELD_UX) out[(slot++) * N + c] = double(ux);
    if (mask & LBM_FIELD_UY) out[(slot++) * N + c] = double(uy);
    if (mask & LBM_FIELD_P) out[(slot++) * N + c] = p;
    if (M == 1 && (mask & LBM_FIELD_RHO)) out[(slot++) * N + c] = 1.0 + double(d);
}

// ---- Remark 4 scheme (on the Remark 3 model) ----
template <typename R>
__device__ __forceinline__ void sp4_u(const R f[kQ], R& ux, R& uy) {
    R jx = R(0), jy = R(0);
#pragma unroll
    for (int i = 1; i < kQ; ++i) {
        if (sx(i)) jx += sx(i) > 0 ? f[i] : -f[i];
        if (sy(i)) jy += sy(i) > 0 ? f[i] : -f[i];
    }
    ux = jx;
    uy = jy;
}

template <typename R>
__device__ __forceinline__ void sp4_force(const SpConst& K, R ux, R uy, R& Fx, R& Fy) {
    const R k = R(K.dl) + R(K.dq) * sqrt(ux * ux + uy * uy);
    Fx = R(K.fx) - k * ux;
    Fy = R(K.fy) - k * uy;
}

// G_i of Remark 3 with force F at velocity u, direction i
template <typename R>
__device__ __forceinline__ R sp4_G(const SpConst& K, int i, R S, R ux, R uy, R Fx, R Fy) {
    const R cu = R(sx(i)) * ux + R(sy(i)) * uy, cF = R(sx(i)) * Fx + R(sy(i)) * Fy;
    const R c2 = R(sx(i) * sx(i) + sy(i) * sy(i));
    return R(sw(i)) * (S + R(3) * cF + R(9) * cu * cF - R(3) * (ux * Fx + uy * Fy) +
                       R(4.5) * (c2 - R(2.0 / 3.0)) * R(K.Qc) * S);
}

template <typename R>
__global__ void sp4_fields_kernel(const R* __restrict__ f, const R* __restrict__ src, long long N, SpConst K,
                                  unsigned mask, double* __restrict__ out) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    R fc[kQ], ux, uy, Fx, Fy;
#pragma unroll
    for (int i = 0; i < kQ; ++i) fc[i] = f[i * N + c];
    sp4_u(fc, ux, uy);
    sp4_force(K, ux, uy, Fx, Fy);
    R rest = R(0);
#pragma unroll
    for (int i = 1; i < kQ; ++i) rest += fc[i];
    const R G0 = sp4_G(K, 0, src[c], ux, uy, Fx, Fy);
    const R p = R(0.6) * (rest - R(2.0 / 3.0) * (ux * ux + uy * uy) + R(K.tau) * G0);
    int slot = 0;
    if (mask & LBM_FIELD_UX) out[(slot++) * N + c] = double(ux);
    if (mask & LBM_FIELD_UY) out[(slot++) * N + c] = double(uy);
    if (mask & LBM_FIELD_P) out[(slot++) * N + c] = double(p);
}

// populations g_i = stored + w_i, widened to FP64
template <typename R>
__global__ void sp1_widen_kernel(const R* __restrict__ in, double* __restrict__ out, long long N, double a0) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
#pragma unroll
    for (int i = 0; i < kQ; ++i) out[i * N + c] = double(in[i * N + c]) + sw(i) * a0;
}

template <typename R>
__global__ void sp_fields_kernel(const R* __restrict__ g, const R* __restrict__ src, long long N, SpConst K,
                                 unsigned mask, double* __restrict__ out) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    R gc[kQ], G[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) gc[i] = g[i * N + c];
    const SpCell<R> m = sp_moments(K, gc, src[c], G);
    int slot = 0;
    if (mask & LBM_FIELD_UX) out[(slot++) * N + c] = double(m.ux);
    if (mask & LBM_FIELD_UY) out[(slot++) * N + c] = double(m.uy);
    if (mask & LBM_FIELD_P) out[(slot++) * N + c] = double(m.p);
}

template <typename R>
__global__ void sp_convert_kernel(const double* __restrict__ in, R* __restrict__ out, long long n) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n) out[c] = R(in[c]);
}

template <typename R>
__global__ void sp_widen_kernel(const R* __restrict__ in, double* __restrict__ out, long long n) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n) out[c] = double(in[c]);
}

// ---- The step ----
// One cell of a unit: float or double with explicit roundings; F2 is a unit of two
// cells (x, x + 1), x even, in packed FP32 instructions (nx even).
template <typename T>
struct One {
    T v;
    One() = default;
    __device__ __forceinline__ One(T x) : v(x) {}
};
__device__ __forceinline__ One<float> operator+(One<float> a, One<float> b) { return __fadd_rn(a.v, b.v); }
__device__ __forceinline__ One<float> operator-(One<float> a, One<float> b) { return __fsub_rn(a.v, b.v); }
__device__ __forceinline__ One<float> operator*(One<float> a, One<float> b) { return __fmul_rn(a.v, b.v); }
__device__ __forceinline__ One<float> fmadd(One<float> a, One<float> b, One<float> c) { return __fmaf_rn(a.v, b.v, c.v); }
__device__ __forceinline__ One<double> operator+(One<double> a, One<double> b) { return __dadd_rn(a.v, b.v); }
__device__ __forceinline__ One<double> operator-(One<double> a, One<double> b) { return __dsub_rn(a.v, b.v); }
__device__ __forceinline__ One<double> operator*(One<double> a, One<double> b) { return __dmul_rn(a.v, b.v); }
__device__ __forceinline__ One<double> fmadd(One<double> a, One<double> b, One<double> c) { return __fma_rn(a.v, b.v, c.v); }
// 1/x and sqrt(x), correctly rounded per lane
template <typename T> __device__ __forceinline__ One<T> sp_inv(One<T> x) { return One<T>(T(1) / x.v); }
template <typename T> __device__ __forceinline__ One<T> sp_sqrt(One<T> x) { return One<T>(sqrt(x.v)); }
__device__ __forceinline__ F2 sp_inv(F2 x) { return F2(1.f / x.v.x, 1.f / x.v.y); }
__device__ __forceinline__ F2 sp_sqrt(F2 x) { return F2(sqrtf(x.v.x), sqrtf(x.v.y)); }

// How a unit sits in memory: T values of one cell or a pair, one access.
template <typename V> struct Unit;
template <typename T> struct Unit<One<T>> {
    using R = T;       // element of a plane
    using E = T;       // a unit in shared memory
    static constexpr int cells = 1;
    __device__ __forceinline__ static One<T> ld(const T* p) { return One<T>(*p); }
    __device__ __forceinline__ static void st(T* p, One<T> v) { *p = v.v; }
    __device__ __forceinline__ static E pack(One<T> v) { return v.v; }
    // the unit dx cells right of unit t of a row in shared memory
    __device__ __forceinline__ static One<T> at(const E* row, int t, int dx) { return One<T>(row[t + dx]); }
    // push direction c_x = dx of unit x of a row; nx: columns
    __device__ __forceinline__ static void push(T* row, int x, int nx, int dx, One<T> v) {
        const int X = x + dx;
        row[X < 0 ? nx - 1 : (X == nx ? 0 : X)] = v.v;
    }
};
template <> struct Unit<F2> {
    using R = float;
    using E = float2;
    static constexpr int cells = 2;
    __device__ __forceinline__ static F2 ld(const float* p) { return F2(*reinterpret_cast<const float2*>(p)); }
    __device__ __forceinline__ static void st(float* p, F2 v) { *reinterpret_cast<float2*>(p) = v.v; }
    __device__ __forceinline__ static E pack(F2 v) { return v.v; }
    __device__ __forceinline__ static F2 at(const E* row, int t, int dx) {
        if (dx < 0) return F2(row[t - 1].y, row[t].x);
        if (dx > 0) return F2(row[t].y, row[t + 1].x);
        return F2(row[t]);
    }
    __device__ __forceinline__ static void push(float* row, int x, int nx, int dx, F2 v) {
        if (dx == 0) {   // keeps the pair together
            st(row + x, v);
        } else {
            row[dx < 0 ? (x == 0 ? nx - 1 : x - 1) : x + 1] = v.v.x;
            row[dx < 0 ? x : (x + 2 == nx ? 0 : x + 2)] = v.v.y;
        }
    }
};

// Constants of the step in the arithmetic type, derived on the host (SpConst) so
// that the kernels convert and combine nothing. F is in the units of g (Remark 2:
// p_0 F_1); ka, kd, k0: 1 + 4.5 (|c|^2 - 2/3) Q of the axes, the diagonals and the
// rest direction (Remark 3), times w_i.
template <typename T>
struct SpK {
    int nx, ny, walls;
    T om, sg, om_h;            // 1/tau_g, 1 - 1/(2 tau_g), om / 2
    T fx, fy, hfx, hfy;        // F, F / 2
    T sgfx, sgfy, hsgfx, hsgfy;   // sg F, sg F / 2
    T ka, kd, k0, ska, skd, sk0;  // Remark 3, Remark 4; s..: times sg
    T tgm, tau;
    T sc, hS, p0, ip0;         // Remarks 1, 2: units of S; S / 2 in them; p_0, 1 / p_0 (Remark 1: unused)
    T q, q0;                   // gs Q = (a q + q0) 12 div u
    T dl, dq;                  // drag
};

template <typename T>
SpK<T> sp_consts(const SpConst& K, int model) {
    SpK<T> k;
    const double sc = model == 2 ? K.p0 : 1.0, fx = sc * K.fx, fy = sc * K.fy, om = K.inv_tau, sg = K.src;
    const double ka = (1.0 + 1.5 * K.Qc) / 9.0, kd = (1.0 + 6.0 * K.Qc) / 36.0, k0 = (1.0 - 3.0 * K.Qc) * 4.0 / 9.0;
    k.nx = K.nx; k.ny = K.ny; k.walls = K.walls;
    k.om = T(om); k.sg = T(sg); k.om_h = T(0.5 * om);
    k.fx = T(fx); k.fy = T(fy); k.hfx = T(0.5 * fx); k.hfy = T(0.5 * fy);
    k.sgfx = T(sg * fx); k.sgfy = T(sg * fy); k.hsgfx = T(0.5 * sg * fx); k.hsgfy = T(0.5 * sg * fy);
    k.ka = T(ka); k.kd = T(kd); k.k0 = T(k0); k.ska = T(sg * ka); k.skd = T(sg * kd); k.sk0 = T(sg * k0);
    k.tgm = T(K.tgm); k.tau = T(K.tau);
    k.sc = T(sc); k.hS = T(0.5 * sc); k.p0 = T(K.p0); k.ip0 = T(K.ip0);
    k.q = T(sg / 36.0); k.q0 = T(sg * K.Qd0 / 12.0);
    k.dl = T(K.dl); k.dq = T(K.dq);
    return k;
}

// The four models by one number: Remarks 1, 2, 3 and the Remark 4 scheme.
// What a cell's neighbours need of it (values of the shared-memory ring): u for
// div u (Remarks 1, 2), G_1 .. G_8 for G_i at x + c_i (Remark 4), nothing (3).
template <int KIND> constexpr int kRing = KIND == 4 ? 8 : (KIND == 3 ? 0 : 2);

// A cell's own values besides its populations and S.
template <typename V>
struct SpMom { V ux, uy, a, b; };   // u; Remarks 1, 2: d and a of the equilibrium; Remark 4: a = G_0

template <typename V>
__device__ __forceinline__ void sp_j(const V (&g)[kQ], V& jx, V& jy) {
    const V a = g[5] - g[7], b = g[6] - g[8];
    jx = (g[1] - g[3]) + (a - b);
    jy = (g[2] - g[4]) + (a + b);
}
template <typename V>
__device__ __forceinline__ V sp_rest(const V (&g)[kQ]) {
    return ((g[1] + g[2]) + (g[3] + g[4])) + ((g[5] + g[6]) + (g[7] + g[8]));
}

// (1 - om) g + x. In FP32 as x - om g, then + g: 1 - om rounded to FP32 would
// give every step a bias of up to 2^-25 of the momentum. (FP64: one operation.)
template <typename T>
__device__ __forceinline__ One<T> sp_relax(T om, One<T> g, One<T> x) {
    if constexpr (sizeof(T) == 8) return fmadd(One<T>(T(1) - om), g, x);
    else return fmadd(One<T>(-om), g, x) + g;
}
__device__ __forceinline__ F2 sp_relax(float om, F2 g, F2 x) { return fmadd(F2(-om), g, x) + g; }
// The odd parts 3 w_i c.T of a vector T over the axes (a) and, as components, the
// diagonals (d = a / 4), from T / 2. The FP32 constants here and below (w_i, w_0 -
// 1, 3/5 and 3 p from p) are the roundings of the remarks' own factors: products
// of them rounded once instead, or sums that conserve the momentum exactly, are
// closer to FP64 but drift from these by up to 1e-4 of a weak velocity component
// in 200 steps.
template <typename V>
__device__ __forceinline__ void sp_odd(V half, V& a, V& d) {
    using T = typename Unit<V>::R;
    a = V(T(1) / T(9)) * (V(T(6)) * half);
    d = V(T(0.25)) * a;
}

// Remark 4: F(u), and the parts of G_i even and odd in c of the pairs (1, 3),
// (2, 4), (5, 7), (6, 8); G_0 returned.
template <typename V, typename T>
__device__ __forceinline__ void sp4_F(const SpK<T>& K, V ux, V uy, V& Fx, V& Fy) {
    const V k = fmadd(V(K.dq), sp_sqrt(fmadd(ux, ux, uy * uy)), V(K.dl));
    Fx = V(K.fx) - k * ux;
    Fy = V(K.fy) - k * uy;
}
template <typename V, typename T>
__device__ __forceinline__ V sp4_Gs(const SpK<T>& K, V S, V ux, V uy, V Fx, V Fy, V (&e)[4], V (&o)[4]) {
    const V t = V(T(-3)) * fmadd(ux, Fx, uy * Fy);
    const V ea = fmadd(S, V(K.ka), V(T(1) / T(9)) * t), ed = fmadd(S, V(K.kd), V(T(1) / T(36)) * t);
    const V up = V(T(0.25)) * (ux + uy), um = V(T(0.25)) * (uy - ux), Fp = Fx + Fy, Fm = Fy - Fx;
    e[0] = fmadd(ux, Fx, ea);
    e[1] = fmadd(uy, Fy, ea);
    e[2] = fmadd(up, Fp, ed);
    e[3] = fmadd(um, Fm, ed);
    V dx, dy;
    sp_odd(V(T(0.5)) * Fx, o[0], dx);
    sp_odd(V(T(0.5)) * Fy, o[1], dy);
    o[2] = dx + dy;
    o[3] = dy - dx;
    return fmadd(S, V(K.k0), V(T(4) / T(9)) * t);
}

// u and what the neighbours need (put(r, value): ring value r).
template <int KIND, typename V, typename T, typename Put>
__device__ __forceinline__ void sp_moments_of(const SpK<T>& K, const V (&g)[kQ], V S, SpMom<V>& m, Put&& put) {
    V jx, jy;
    sp_j(g, jx, jy);
    if constexpr (KIND == 1) {                       // rho - 1 (Eq. 27aa), rho; u (Eq. 27a)
        m.a = fmadd(V(K.hS), S, g[0] + sp_rest(g));
        m.b = V(T(1)) + m.a;
        const V ir = sp_inv(m.b);
        m.ux = (jx + V(K.hfx)) * ir;
        m.uy = (jy + V(K.hfy)) * ir;
    } else if constexpr (KIND == 2) {                // p - p_0, p_0
        m.a = fmadd(V(K.hS), S, g[0] + sp_rest(g));
        m.b = V(K.p0);
        m.ux = (jx + V(K.hfx)) * V(K.ip0);
        m.uy = (jy + V(K.hfy)) * V(K.ip0);
    } else if constexpr (KIND == 3) {
        m.ux = jx + V(K.hfx);
        m.uy = jy + V(K.hfy);
    } else {                                         // Remark 4: u = sum c f, G_i with F(u)
        m.ux = jx;
        m.uy = jy;
        V Fx, Fy, e[4], o[4];
        sp4_F(K, jx, jy, Fx, Fy);
        m.a = sp4_Gs(K, S, jx, jy, Fx, Fy, e, o);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            put(pair2(k) - 1, e[k] + o[k]);
            put(sopp(pair2(k)) - 1, e[k] - o[k]);
        }
    }
    if constexpr (KIND == 1 || KIND == 2) {
        put(0, m.ux);
        put(1, m.uy);
    }
}

// Collision (Eq. 24 with the remark's equilibrium and force term). Opposite
// directions share the part even in c: with sg = 1 - 1/(2 tau_g) and om = 1/tau_g,
//   g_i* = (1 - om) g_i + E_i +- O_i,  E_i = (c.u)(c.V) + E0,  O_i = 3 w_i c.T,
// V = w_i (4.5 (om a [- sg S]) u + 9 sg F), T = om a u + sg F; the axes' weights
// are four times the diagonals'. nb(r, dx, dy): ring value r of a
// neighbour (mirrored about a wall); up: u at t - 1 (Remark 4); emit(i, value,
// wall value): the population leaving in direction i, and what returns if a wall
// reflects it (the same but for Remark 4).
template <int KIND, typename V, typename T, typename Nb, typename Emit>
__device__ __forceinline__ void sp_collide(const SpK<T>& K, const V (&g)[kQ], V S, const SpMom<V>& m, V upx, V upy,
                                           Nb&& nb, Emit&& emit) {
    const V ux = m.ux, uy = m.uy;
    const V uu = fmadd(ux, ux, uy * uy);
    const V ninth(T(1) / T(9)), q(T(0.25));
    if constexpr (KIND == 4) {
        const V G0 = m.a;
        V Px, Py, pe[4], po[4];
        sp4_F(K, upx, upy, Px, Py);
        const V P0 = sp4_Gs(K, S, upx, upy, Px, Py, pe, po);
        // Eq. 28 for the unshifted f: p = 3/5 [sum f_i - (2/3) u.u + tau_g G_0]
        const V p3 = V(T(3)) * (V(T(0.6)) * fmadd(V(K.tau), G0, fmadd(V(T(-2) / T(3)), uu, sp_rest(g))));
        const V om(K.om), half(T(0.5));
        const V uu15 = V(T(-1.5)) * uu, b = p3 + uu15;   // 3 p - 1.5 u.u
        const V geq0 = fmadd(V(T(4.0 / 9.0 - 1.0)), p3, V(T(4) / T(9)) * uu15);
        emit(0, sp_relax(K.om, g[0], fmadd(om, geq0, fmadd(half, G0 - P0, G0))), V(T(0)));
        const V ga = ninth * b, gd = q * ga;
        const V up = q * (ux + uy), um = q * (uy - ux);
        const V hx = half * ux, hy = half * uy;
        const V ge[4] = {fmadd(hx, ux, ga), fmadd(hy, uy, ga), fmadd(V(T(2)) * up, up, gd),
                         fmadd(V(T(2)) * um, um, gd)};
        V ax, ay, dx, dy;
        sp_odd(hx, ax, dx);
        sp_odd(hy, ay, dy);
        const V go[4] = {ax, ay, dx + dy, dy - dx};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = pair2(k), j = sopp(i);
            // om g^eq_i - G_i(t - 1) / 2, even and odd parts
            const V A = fmadd(om, ge[k], V(T(-0.5)) * pe[k]), B = fmadd(om, go[k], V(T(-0.5)) * po[k]);
            const V Gi = nb(i - 1, 0, 0), Gj = nb(j - 1, 0, 0);
            const V ni = nb(i - 1, sx(i), sy(i)), nj = nb(j - 1, sx(j), sy(j));
            // without G_i(x + c_i) / 2
            const V pi = sp_relax(K.om, g[i], Gi + (A + B)), pj = sp_relax(K.om, g[j], Gj + (A - B));
            // bounce-back of f - G/2: leaves with G_i(x + c_i) / 2 less, returns as opp(i) with G_opp(x) / 2
            emit(i, fmadd(half, ni, pi), fmadd(half, Gj, pi));
            emit(j, fmadd(half, nj, pj), fmadd(half, Gi, pj));
        }
        return;
    } else {
        V Vx, Vy, Tx, Ty, Ea, Ed, r0;   // Tx, Ty: (om a u + sg F) / 2
        const V uF = fmadd(ux, V(K.fx), uy * V(K.fy));
        if constexpr (KIND == 3) {
            // Eq. 28: p = 3/5 [sum g_i + S/2 - (2/3) u.u + (tau_g - 1/2) G_0]
            const V t = V(T(-3)) * uF;
            const V G0 = fmadd(S, V(K.k0), V(T(4) / T(9)) * t);
            const V p3 = V(T(3)) * (V(T(0.6)) * fmadd(V(K.tgm), G0, fmadd(V(T(-2) / T(3)), uu,
                                                                          fmadd(V(T(0.5)), S, sp_rest(g)))));
            const V omp = V(K.om) * p3;
            const V b0 = fmadd(V(K.om), V(T(-1.5)) * uu, V(K.sg) * t), b = omp + b0;
            Vx = fmadd(V(K.om_h), ux, V(K.sgfx));
            Vy = fmadd(V(K.om_h), uy, V(K.sgfy));
            Tx = fmadd(V(K.om_h), ux, V(K.hsgfx));
            Ty = fmadd(V(K.om_h), uy, V(K.hsgfy));
            Ea = fmadd(S, V(K.ska), ninth * b);
            Ed = fmadd(S, V(K.skd), V(T(1) / T(36)) * b);
            r0 = fmadd(V(T(4.0 / 9.0 - 1.0)), omp, fmadd(S, V(K.sk0), V(T(4) / T(9)) * b0));
        } else {
            // 12 div u (Eq. 30a)
            const V sa = nb(0, 1, 1) - nb(0, -1, -1), sb = nb(0, -1, 1) - nb(0, 1, -1);
            const V ta = nb(1, 1, 1) - nb(1, -1, -1), tb = nb(1, -1, 1) - nb(1, 1, -1);
            const V ax = nb(0, 1, 0) - nb(0, -1, 0), ay = nb(1, 0, 1) - nb(1, 0, -1);
            const V div = fmadd(V(T(4)), ax + ay, (sa - sb) + (ta + tb));
            const V gq = fmadd(m.b, V(K.q), V(K.q0)) * div;          // sg Q div u
            const V Sg = V(K.sc) * S, om(K.om), sg(K.sg);
            const V h = V(K.om_h) * m.b;                              // om a / 2
            V hA, S2;
            if constexpr (KIND == 1) {                                // with the u u S of Remark 1
                hA = h - V(T(0.5)) * (sg * Sg);
                S2 = fmadd(V(T(1.5)) * uu, Sg, Sg);
            } else {
                hA = h;
                S2 = Sg;
            }
            Vx = fmadd(hA, ux, V(K.sgfx));
            Vy = fmadd(hA, uy, V(K.sgfy));
            if constexpr (KIND == 2) {   // (om p_0 / 2, a constant, rounded would be a bias of every step)
                Tx = fmadd(V(K.om_h), m.b * ux, V(K.hsgfx));
                Ty = fmadd(V(K.om_h), m.b * uy, V(K.hsgfy));
            } else {
                Tx = fmadd(h, ux, V(K.hsgfx));
                Ty = fmadd(h, uy, V(K.hsgfy));
            }
            const V b = fmadd(om, fmadd(V(T(-1.5)) * m.b, uu, m.a), sg * fmadd(V(T(-3)), uF, S2));
            Ea = ninth * fmadd(V(T(1.5)), gq, b);
            Ed = V(T(1) / T(36)) * fmadd(V(T(6)), gq, b);
            r0 = V(T(4) / T(9)) * fmadd(V(T(-3)), gq, b);
        }
        auto out = [&](int i, V v) { emit(i, v, v); };
        out(0, sp_relax(K.om, g[0], r0));
        auto pair = [&](int i, int j, V E, V O) {
            out(i, sp_relax(K.om, g[i], E + O));
            out(j, sp_relax(K.om, g[j], E - O));
        };
        V ox, oy, dx, dy;
        sp_odd(Tx, ox, dx);
        sp_odd(Ty, oy, dy);
        pair(1, 3, fmadd(ux, Vx, Ea), ox);
        pair(2, 4, fmadd(uy, Vy, Ea), oy);
        pair(5, 7, fmadd(q * (ux + uy), Vx + Vy, Ed), dx + dy);
        pair(6, 8, fmadd(q * (uy - ux), Vy - Vx, Ed), dy - dx);
    }
}

// Push-streaming of a unit at column x of row y: into its neighbours, or back
// reversed from a wall (halfway bounce-back). 32-bit offsets: 9 nx ny < 2^31.
template <typename V>
struct SpPush {
    using U = Unit<V>;
    typename U::R* out;
    int N, nx, x, y, up, dn;
    bool bot, top;
    template <typename T>
    __device__ __forceinline__ SpPush(const SpK<T>& K, typename U::R* out_, int N_, int x_, int y_)
        : out(out_), N(N_), nx(K.nx), x(x_), y(y_) {
        bot = K.walls && y == 0;
        top = K.walls && y == K.ny - 1;
        dn = y == 0 ? K.ny - 1 : y - 1;   // (not used at a wall)
        up = y == K.ny - 1 ? 0 : y + 1;
    }
    __device__ __forceinline__ void operator()(int i, V v, V w) const {
        if ((sy(i) > 0 && top) || (sy(i) < 0 && bot)) {
            U::st(out + sopp(i) * N + y * nx + x, w);
            return;
        }
        U::push(out + i * N + (sy(i) == 0 ? y : (sy(i) > 0 ? up : dn)) * nx, x, nx, sx(i), v);
    }
};

// Remark 3, large domains: nothing of a neighbour is needed, one unit a thread.
// 4096 x 4096 FP32 186 us a step (1.0 of the copy bandwidth); FP64 bound by its
// FP64 operations: 2048 x 2048 1235 -> 638 us with the opposite pairs' even and odd
// parts.
template <typename V>
__global__ void __launch_bounds__(256, 4) sp_cell_kernel(const typename Unit<V>::R* __restrict__ gin,
                                                      typename Unit<V>::R* __restrict__ gout,
                                                      const typename Unit<V>::R* __restrict__ src, int N,
                                                      SpK<typename Unit<V>::R> K) {
    using U = Unit<V>;
    const int c = U::cells * (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (c >= N) return;
    const int y = c / K.nx, x = c - y * K.nx;
    V g[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) g[i] = U::ld(gin + i * N + c);
    const V S = U::ld(src + c);
    SpMom<V> m;
    sp_moments_of<3>(K, g, S, m, [](int, V) {});
    sp_collide<3>(K, g, S, m, V(), V(), [](int, int, int) { return V(); }, SpPush<V>(K, gout, N, x, y));
}

// ---- One pass a step: row marches of Remarks 1, 2 and 4 ----
// These models couple a cell to its neighbours only through functions of the
// neighbours' own populations (u in div u; G_i at x + c_i), so a step is one
// kernel: a block owns a strip of columns and marches over a run of rows, keeping
// what the neighbours need of three rows in a shared-memory ring and the
// populations of the collision row and the next one in registers. Per row: the
// loads of the row after the next are issued, the next row's ring values formed,
// one barrier, the collision. Every population is read once: in FP32 76 bytes a
// cell for Remarks 1 and 2 (two kernels, one writing u, moved 132), 92 for Remark
// 4 (160: of t - 1 it keeps u, two planes updated in place, and forms F(u) again).
// 4096 x 4096 FP32, two kernels -> here, us a step: Remark 1 375 -> 206 (0.91 of
// the copy bandwidth), 2 330 -> 217, 4 489 -> 309 (0.74: three quarters of it
// arithmetic at 16 warps a SM); 2048 x 2048 FP64 (half the FP64 operations) 1790 ->
// 878, 1525 -> 780, 2459 -> 1691.
//
// Thread t holds unit t - 1 of the strip [x0, x0 + w): the first and the last hold
// one unit of halo, which they only prepare. Neighbouring runs march in opposite
// directions, so that the rows both need at a shared boundary are read together.
struct SpRun {
    int rows, strips, w;   // rows a run, strips of w columns
};
struct SpMarch {   // the block's run: Y0 its first row, d its direction, n its rows
    int x0, wc, Y0, d, n, ny, walls;
    template <typename T>
    __device__ __forceinline__ SpMarch(const SpK<T>& K, const SpRun& r) : ny(K.ny), walls(K.walls) {
        const int run = blockIdx.x / r.strips, strip = blockIdx.x - run * r.strips;
        x0 = strip * r.w;
        wc = min(r.w, K.nx - x0);
        const int ya = run * r.rows, yb = min(ny, ya + r.rows);
        n = yb - ya;
        d = (run & 1) ? 1 : -1;
        Y0 = d > 0 ? ya : yb - 1;
    }
    __device__ __forceinline__ bool ghost(int y) const { return walls && (y < 0 || y >= ny); }
    __device__ __forceinline__ int row(int y) const { return y < 0 ? y + ny : (y >= ny ? y - ny : y); }
    __device__ __forceinline__ static int slot(int y) { return (y + 4) & 3; }
    // ring slot of row y + r as row y's stencil sees it: the wall mirrors it onto y
    __device__ __forceinline__ int near(int y, int r) const { return slot(ghost(y + r) ? y : y + r); }
};

constexpr int kSpThreads = 128;   // most threads of a march block, all of a tile block

template <int KIND, typename V, int OCC>
__global__ void __launch_bounds__(kSpThreads, OCC) sp_march_kernel(const typename Unit<V>::R* __restrict__ gin,
                                                                   typename Unit<V>::R* __restrict__ gout,
                                                                   const typename Unit<V>::R* __restrict__ src,
                                                                   typename Unit<V>::R* __restrict__ uprev, int N,
                                                                   SpK<typename Unit<V>::R> K, SpRun run) {
    using U = Unit<V>;
    __shared__ typename U::E ring[4][kRing<KIND>][kSpThreads];
    const SpMarch A(K, run);
    const int t = threadIdx.x, nx = K.nx;
    const bool in = U::cells * t < A.wc + 2 * U::cells, own = t >= 1 && U::cells * t < A.wc + U::cells;
    int x = A.x0 + U::cells * (t - 1);
    x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
    auto load = [&](int y, V (&g)[kQ], V& S) {
        if (!in || A.ghost(y)) return;
        const int c = A.row(y) * nx + x;
#pragma unroll
        for (int i = 0; i < kQ; ++i) g[i] = U::ld(gin + i * N + c);
        S = U::ld(src + c);
    };
    auto prepare = [&](int y, const V (&g)[kQ], V S, SpMom<V>& m) {
        if (!in || A.ghost(y)) return;
        auto& slot = ring[A.slot(y)];
        sp_moments_of<KIND>(K, g, S, m, [&](int r, V v) { slot[r][t] = U::pack(v); });
    };
    V g[kQ], S, gn[kQ], Sn;
    SpMom<V> m, mn;
    load(A.Y0 - A.d, gn, Sn);
    load(A.Y0, g, S);
    prepare(A.Y0 - A.d, gn, Sn, mn);
    prepare(A.Y0, g, S, m);
    load(A.Y0 + A.d, gn, Sn);
    for (int k = 0; k < A.n; ++k) {
        const int y = A.Y0 + k * A.d, c = y * nx + x;
        V upx, upy;
        if (KIND == 4 && own) {
            upx = U::ld(uprev + c);
            upy = U::ld(uprev + N + c);
        }
        prepare(y + A.d, gn, Sn, mn);
        V gx[kQ], Sx;
        if (k + 1 < A.n) load(y + 2 * A.d, gx, Sx);
        __syncthreads();
        if (own) {
            if constexpr (KIND == 4) {
                U::st(uprev + c, m.ux);
                U::st(uprev + N + c, m.uy);
            }
            sp_collide<KIND>(K, g, S, m, upx, upy,
                             [&](int r, int dx, int dy) { return U::at(ring[A.near(y, dy)][r], t, dx); },
                             SpPush<V>(K, gout, N, x, y));
        }
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            g[i] = gn[i];
            gn[i] = gx[i];
        }
        S = Sn;
        Sn = Sx;
        m = mn;
    }
}

// ---- Small domains: several steps in one cooperative launch over tiles ----
// As step_kernel_tile (lbm_tile.cuh): tiles of at most 128 units, all rows at
// once, an item's step waiting only for the items within 3 cells. Up to where the
// marches above fill the GPU, a launch a step costs more than the step.
struct SpTileArgs {
    const void *g0, *g1;   // buffer sets: step s reads g0 when s is even
    const void* src;
    void* uprev;
    int N, nitems, nsteps, ulog, wait_limit;
    const lbm::WorkItem* work;
    const int* nbr;
    int *done, *status;
};

template <int KIND, typename V, int OCC>
__global__ void __launch_bounds__(kSpThreads, OCC) sp_tile_kernel(const SpTileArgs a, SpK<typename Unit<V>::R> K) {
    using U = Unit<V>;
    using R = typename U::R;
    // (2^u + 2) x (rows + 2) units: at most 34 x 6 over the shapes 2^u x 128 / 2^u
    constexpr int NR = kRing<KIND> > 0 ? kRing<KIND> : 1;
    __shared__ typename U::E ring[NR][208];
    __shared__ int s_bad;
    const int tid = threadIdx.x, nx = K.nx, ny = K.ny, N = a.N;
    const int W = (1 << a.ulog) + 2;
    const R* src = static_cast<const R*>(a.src);
    R* uprev = static_cast<R*>(a.uprev);
    for (int s = 0; s < a.nsteps; ++s) {
        const R* gin = static_cast<const R*>((s & 1) ? a.g1 : a.g0);
        R* gout = static_cast<R*>(const_cast<void*>((s & 1) ? a.g0 : a.g1));
        for (int item = blockIdx.x; item < a.nitems; item += gridDim.x) {
            const lbm::WorkItem wk = a.work[item];
            if (s > 0 && !lbm::tile_wait(a.done, a.nbr + item * lbm::kMaxTileNbr, s, a.wait_limit, a.status,
                                         a.done + a.nitems, &s_bad, tid))
                return;
            const int nu = wk.dir / U::cells, rows = wk.nrows;
            const int tx = tid & (W - 3), ty = tid >> a.ulog;
            const bool act = tx < nu && ty < rows;
            auto prepare = [&](int ry, int rx, V (&g)[kQ], V& S, SpMom<V>& m) {   // unit rx of row ry, from -1
                int x = wk.x0 + rx * U::cells, y = wk.ystart + ry;
                x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
                if (K.walls) y = y < 0 ? 0 : (y >= ny ? ny - 1 : y);   // the wall mirrors its row
                else y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
                const int c = y * nx + x, at = (ry + 1) * W + rx + 1;
#pragma unroll
                for (int i = 0; i < kQ; ++i) g[i] = U::ld(gin + i * N + c);
                S = U::ld(src + c);
                sp_moments_of<KIND>(K, g, S, m, [&](int r, V v) { ring[r][at] = U::pack(v); });
            };
            V g[kQ], S, upx, upy;
            SpMom<V> m;
            const int x = wk.x0 + tx * U::cells, y = wk.ystart + ty, c = y * nx + x;
            if (act) {
                if (KIND == 4) {
                    upx = U::ld(uprev + c);
                    upy = U::ld(uprev + N + c);
                }
                prepare(ty, tx, g, S, m);
            }
            if constexpr (KIND != 3) {
                const int ownth = rows << a.ulog, halo = 2 * (nu + 2) + 2 * rows;
                for (int k = tid >= ownth ? tid - ownth : tid + kSpThreads - ownth; k < halo; k += kSpThreads) {
                    const int cap = 2 * (nu + 2), q = k - cap;
                    const int ry = k < cap ? (k < nu + 2 ? -1 : rows) : q >> 1;
                    const int rx = k < cap ? (k < nu + 2 ? k : k - nu - 2) - 1 : ((q & 1) ? nu : -1);
                    V gh[kQ], Sh;
                    SpMom<V> mh;
                    prepare(ry, rx, gh, Sh, mh);
                }
                __syncthreads();
            }
            if (act) {
                if constexpr (KIND == 4) {
                    U::st(uprev + c, m.ux);
                    U::st(uprev + N + c, m.uy);
                }
                const int at = (ty + 1) * W + tx + 1;
                sp_collide<KIND>(K, g, S, m, upx, upy,
                                 [&](int r, int dx, int dy) { return U::at(ring[r], at + dy * W, dx); },
                                 SpPush<V>(K, gout, N, x, y));
            }
            __syncthreads();   // every thread's stores of the step issued, the ring free
            if (tid == 0 && a.nsteps > 1) {
                __threadfence();
                atomicExch(a.done + item, s + 1);
            }
        }
    }
}

}  // namespace

struct lbm_sp_ctx {
    lbm_sp_params p;
    int form = 0;                      // LBM_F64 or LBM_F32
    long long N = 0;
    void* g[2] = {nullptr, nullptr};
    void* src = nullptr;
    void* ufield = nullptr;            // Remark 4 scheme: u of the step before (2 planes)
    double* d_tmp = nullptr;           // staging for inputs and outputs
    int cur = 0;
    bool ready = false;
    long long time = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    SpConst K{};
    SpK<float> kf;                     // the step's constants in the arithmetic type
    SpK<double> kd;
    int kind = 3;                      // 1, 2, 3: Remarks; 4: the Remark 4 scheme
    int cells = 1;                     // cells a unit: 2 in FP32 with nx even
    const void* kernel = nullptr;      // one step a launch: row march, Remark 3 one unit a thread
    SpRun run{};
    int threads = kSpThreads;
    const void* tile = nullptr;        // small domains: several steps a launch (null: not taken)
    int tile_items = 0, tile_grid = 0, tile_ulog = 0;
    void* d_tile = nullptr;            // items, neighbours, step counters and abort flag
    lbm::WorkItem* d_tile_work = nullptr;
    int* d_tile_nbr = nullptr;
    int* d_tile_done = nullptr;
    int* d_status = nullptr;           // set by a bounded wait that ran out
    std::string err;
};

namespace {

lbm_status sp_fail(lbm_sp_ctx* c, lbm_status st, const std::string& m) {
    if (c) c->err = m;
    return st;
}
lbm_status sp_cuda(lbm_sp_ctx* c, cudaError_t e, const char* what) {
    return sp_fail(c, LBM_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}
size_t sp_elem(int form) { return form == LBM_F64 ? 8 : 4; }
int blocks(long long n) { return (int)((n + 255) / 256); }

void sp_release(lbm_sp_ctx* c) {
    cudaFree(c->g[0]);
    cudaFree(c->g[1]);
    cudaFree(c->src);
    cudaFree(c->ufield);
    cudaFree(c->d_tile);
    cudaFree(c->d_status);
    cudaFree(c->d_tmp);
    if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
}

// The step kernels of a model for unit type V, and the resident blocks of 128
// threads a SM their registers are sized for. The row march holds two rows of
// populations and a third in flight. Measured at 4096 x 4096, pairs, us a step:
// Remark 1 220 / 206 / 282 with 4 / 5 / 6 blocks, Remark 2 216 / 217 / 235, Remark 4
// 330 / 309 / 367 with 3 / 4 / 5; FP64 the same with 2 to 4 (bound by its FP64
// operations).
template <typename V>
void sp_kernels(int kind, const void** step, const void** tile) {
    constexpr bool f64 = sizeof(typename Unit<V>::R) == 8, pair = Unit<V>::cells == 2;
    constexpr int m = f64 ? 3 : pair ? 5 : 6, m2 = f64 ? 3 : pair ? 4 : 6, m4 = f64 ? 3 : pair ? 4 : 6;
    constexpr int o = f64 ? 3 : pair ? 4 : 6;
    switch (kind) {
        case 1:
            *step = (const void*)sp_march_kernel<1, V, m>;
            *tile = (const void*)sp_tile_kernel<1, V, o>;
            break;
        case 2:
            *step = (const void*)sp_march_kernel<2, V, m2>;
            *tile = (const void*)sp_tile_kernel<2, V, o>;
            break;
        case 4:
            *step = (const void*)sp_march_kernel<4, V, m4>;
            *tile = (const void*)sp_tile_kernel<4, V, o>;
            break;
        default:
            *step = (const void*)sp_cell_kernel<V>;
            *tile = (const void*)sp_tile_kernel<3, V, o>;
    }
}

// Chooses the step kernels and their launch shapes.
lbm_status sp_plan(lbm_sp_ctx* c) {
    c->kind = c->p.scheme == LBM_SP_SCHEME_REMARK4 ? 4
              : c->p.model == LBM_SP_NEARLY_INCOMPRESSIBLE ? 1
              : c->p.model == LBM_SP_HE_INCOMPRESSIBLE ? 2 : 3;
    c->kf = sp_consts<float>(c->K, c->p.model);
    c->kd = sp_consts<double>(c->K, c->p.model);
    c->cells = c->form == LBM_F32 && c->p.nx % 2 == 0 ? 2 : 1;
    if (c->form == LBM_F64) sp_kernels<One<double>>(c->kind, &c->kernel, &c->tile);
    else if (c->cells == 2) sp_kernels<F2>(c->kind, &c->kernel, &c->tile);
    else sp_kernels<One<float>>(c->kind, &c->kernel, &c->tile);
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    auto slots = [&](const void* k, int threads) {
        int occ = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, threads, 0);
        return (long long)sms * (occ > 0 ? occ : 1);
    };
    const int units = c->p.nx / c->cells;
    if (c->kind != 3) {
        // strips of equal width, at most `threads` - 2 units; run lengths for the
        // fewest (waves of resident blocks) x (rows + 2 for the prologue)
        long long best = -1;
        for (int threads = 64; threads <= kSpThreads; threads += 32) {
            const int strips = (units + threads - 3) / (threads - 2), w = (units + strips - 1) / strips;
            const long long target = slots(c->kernel, threads);
            for (int r = 1; r <= c->p.ny; ++r) {
                const int rows = (c->p.ny + r - 1) / r, runs = (c->p.ny + rows - 1) / rows;
                const long long cost = ((long long)strips * runs + target - 1) / target * (rows + 2);
                if (best < 0 || cost < best) {
                    best = cost;
                    c->threads = threads;
                    c->run = SpRun{rows, strips, w * c->cells};
                }
            }
        }
    }
    // Tiles, several steps a launch, while every tile is resident at once (FP64:
    // two rounds): a step of a small domain is the latency of a launch. us a step,
    // tiles and one launch a step: 64 x 64 Remark 1 FP32 3.0 and 4.2, FP64 6.0 and
    // 8.8; 256 x 256 3.7 and 6.2, 18.6 and 26.9; 400 x 400 (3 rounds) 8.7 and 6.2,
    // 50.9 and 49.5.
    auto count = [&](int u, int r) { return (long long)((units + u - 1) / u) * ((c->p.ny + r - 1) / r); };
    int U, R;
    lbm::tile_shape(count, sms, &U, &R);
    const long long tslots = slots(c->tile, kSpThreads);
    if (count(8, 16) < count(U, R) && count(U, R) > tslots) {
        U = 8;
        R = 16;
    }
    if (count(U, R) > (c->form == LBM_F64 ? 2 : 1) * tslots) {
        c->tile = nullptr;
        return LBM_OK;
    }
    lbm::TileList list;
    lbm::add_tiles(list, 0, c->p.nx, c->p.ny, c->cells, c->p.bc_y != LBM_BC_BOUNCEBACK, U, R);
    const size_t wb = (list.items.size() * sizeof(lbm::WorkItem) + 255) & ~size_t(255);
    const size_t nb = (list.nbr.size() * sizeof(int) + 255) & ~size_t(255);
    const size_t db = (list.items.size() + 1) * sizeof(int);
    cudaError_t r = cudaMalloc(&c->d_tile, wb + nb + db);
    if (r != cudaSuccess) return r == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA;
    c->d_tile_work = static_cast<lbm::WorkItem*>(c->d_tile);
    c->d_tile_nbr = reinterpret_cast<int*>(static_cast<char*>(c->d_tile) + wb);
    c->d_tile_done = reinterpret_cast<int*>(static_cast<char*>(c->d_tile) + wb + nb);
    if (cudaMemcpy(c->d_tile_work, list.items.data(), list.items.size() * sizeof(lbm::WorkItem),
                   cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(c->d_tile_nbr, list.nbr.data(), list.nbr.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess)
        return LBM_ECUDA;
    c->tile_items = (int)list.items.size();
    c->tile_grid = (int)(c->tile_items < tslots ? c->tile_items : tslots);
    while ((1 << c->tile_ulog) < U) ++c->tile_ulog;
    return LBM_OK;
}

// Queues one step.
cudaError_t sp_step_once(lbm_sp_ctx* c) {
    const void* in = c->g[c->cur];
    void* out = c->g[1 - c->cur];
    int N = (int)c->N;
    void* k = c->form == LBM_F64 ? (void*)&c->kd : (void*)&c->kf;
    c->cur ^= 1;
    if (c->kind == 3) {
        void* args[] = {&in, &out, &c->src, &N, k};
        return cudaLaunchKernel(c->kernel, dim3(blocks(c->N / c->cells)), dim3(256), args, 0, c->stream);
    }
    void* args[] = {&in, &out, &c->src, &c->ufield, &N, k, &c->run};
    const int runs = (c->p.ny + c->run.rows - 1) / c->run.rows;
    return cudaLaunchKernel(c->kernel, dim3(runs * c->run.strips), dim3(c->threads), args, 0, c->stream);
}

// Queues n steps on tiles as one cooperative launch, after zeroing the step
// counters and the abort flag.
cudaError_t sp_step_tiles(lbm_sp_ctx* c, int n) {
    SpTileArgs a;
    a.g0 = c->g[c->cur];
    a.g1 = c->g[1 - c->cur];
    a.src = c->src;
    a.uprev = c->ufield;
    a.N = (int)c->N;
    a.nitems = c->tile_items;
    a.nsteps = n;
    a.ulog = c->tile_ulog;
    a.wait_limit = lbm::kWaitLimit;
    a.work = c->d_tile_work;
    a.nbr = c->d_tile_nbr;
    a.done = c->d_tile_done;
    a.status = c->d_status;
    if (n > 1) {
        const cudaError_t e = cudaMemsetAsync(a.done, 0, ((size_t)c->tile_items + 1) * sizeof(int), c->stream);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {&a, c->form == LBM_F64 ? (void*)&c->kd : (void*)&c->kf};
    c->cur ^= n & 1;
    // one step: no block waits, so the grid need not be resident at once
    return n > 1 ? cudaLaunchCooperativeKernel(c->tile, dim3(c->tile_grid), dim3(kSpThreads), args, 0, c->stream)
                 : cudaLaunchKernel(c->tile, dim3(c->tile_grid), dim3(kSpThreads), args, 0, c->stream);
}

// After a synchronisation: a bounded wait of the tiles that ran out.
lbm_status sp_device_status(lbm_sp_ctx* c) {
    if (!c->tile) return LBM_OK;
    int st = 0;
    const cudaError_t r = cudaMemcpyAsync(&st, c->d_status, sizeof(int), cudaMemcpyDeviceToHost, c->stream);
    if (r != cudaSuccess || cudaStreamSynchronize(c->stream) != cudaSuccess) return sp_cuda(c, r, "status read-back");
    return st == 0 ? LBM_OK : sp_fail(c, LBM_ETIMEOUT, "a bounded device wait ran out in the step kernel");
}

template <int M>
void sp1_fields(lbm_sp_ctx* c, unsigned mask) {
    if (c->form == LBM_F64)
        sp1_fields_kernel<M, double><<<blocks(c->N), 256, 0, c->stream>>>(
            static_cast<const double*>(c->g[c->cur]), static_cast<const double*>(c->src), c->N, c->K, mask, c->d_tmp);
    else
        sp1_fields_kernel<M, float><<<blocks(c->N), 256, 0, c->stream>>>(
            static_cast<const float*>(c->g[c->cur]), static_cast<const float*>(c->src), c->N, c->K, mask, c->d_tmp);
}

}  // namespace

extern "C" {

lbm_status lbm_sp_create(const lbm_sp_params* params, int precision, void* cuda_stream, lbm_sp_ctx** out) {
    if (!out) return LBM_EINVAL;
    *out = nullptr;
    if (!params) return LBM_EINVAL;
    const lbm_sp_params& p = *params;
    if (p.nx < 3 || p.ny < 3 || (long long)p.nx * p.ny >= (1LL << 31) / 9) return LBM_EINVAL;
    if (p.bc_y != LBM_BC_PERIODIC && p.bc_y != LBM_BC_BOUNCEBACK) return LBM_EINVAL;
    if (p.model != LBM_SP_INCOMPRESSIBLE_SOURCE && p.model != LBM_SP_NEARLY_INCOMPRESSIBLE &&
        p.model != LBM_SP_HE_INCOMPRESSIBLE)
        return LBM_EINVAL;
    if (p.model == LBM_SP_HE_INCOMPRESSIBLE && !(std::isfinite(p.p0) && p.p0 > 0)) return LBM_EINVAL;
    if ((p.scheme != LBM_SP_SCHEME_EQ24 && p.scheme != LBM_SP_SCHEME_REMARK4) || p.reserved != 0) return LBM_EINVAL;
    if (!(std::isfinite(p.drag_lin) && p.drag_lin >= 0) || !(std::isfinite(p.drag_quad) && p.drag_quad >= 0))
        return LBM_EINVAL;
    // a velocity-dependent force makes Eq. 27a implicit: it needs the Remark 4 scheme,
    // which is built on the Remark 3 model
    if (p.scheme == LBM_SP_SCHEME_EQ24 && (p.drag_lin != 0 || p.drag_quad != 0)) return LBM_EINVAL;
    if (p.scheme == LBM_SP_SCHEME_REMARK4 && p.model != LBM_SP_INCOMPRESSIBLE_SOURCE) return LBM_EINVAL;
    if (!(std::isfinite(p.nu) && p.nu > 0) || !(std::isfinite(p.xi) && p.xi >= 0) || !std::isfinite(p.force_x) ||
        !std::isfinite(p.force_y))
        return LBM_EINVAL;
    if (precision != LBM_F64 && precision != LBM_F32) return LBM_EINVAL;
    lbm_sp_ctx* c = new lbm_sp_ctx();
    c->p = p;
    c->form = precision;
    c->N = (long long)p.nx * p.ny;
    const double tau = 3.0 * p.nu + 0.5;
    c->K = SpConst{p.nx, p.ny, p.bc_y == LBM_BC_BOUNCEBACK ? 1 : 0, 1.0 / tau, 1.0 - 0.5 / tau, tau - 0.5,
                   1.0 / 3.0 - p.xi / (tau - 0.5), p.force_x, p.force_y, p.drag_lin, p.drag_quad, p.p0,
                   tau, -p.xi / (tau - 0.5), 0.5 * p.p0, p.p0 > 0 ? 1.0 / p.p0 : 0.0, 0.5 * p.p0 * p.force_x,
                   0.5 * p.p0 * p.force_y};
    const size_t e = sp_elem(precision);
    cudaError_t r;
    if ((r = cudaMalloc(&c->g[0], kQ * c->N * e)) != cudaSuccess ||
        (r = cudaMalloc(&c->g[1], kQ * c->N * e)) != cudaSuccess ||
        (r = cudaMalloc(&c->src, c->N * e)) != cudaSuccess ||
        (p.scheme == LBM_SP_SCHEME_REMARK4 && (r = cudaMalloc(&c->ufield, 2 * c->N * e)) != cudaSuccess) ||
        (r = cudaMalloc((void**)&c->d_status, sizeof(int))) != cudaSuccess ||
        (r = cudaMalloc((void**)&c->d_tmp, kQ * c->N * sizeof(double))) != cudaSuccess) {
        sp_release(c);
        delete c;
        return r == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA;
    }
    if (cuda_stream) {
        c->stream = static_cast<cudaStream_t>(cuda_stream);
    } else if (cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking) == cudaSuccess) {
        c->own_stream = true;
    } else {
        sp_release(c);
        delete c;
        return LBM_ECUDA;
    }
    const lbm_status st = sp_plan(c);
    if (st != LBM_OK) {
        sp_release(c);
        delete c;
        return st;
    }
    *out = c;
    return LBM_OK;
}

lbm_status lbm_sp_init(lbm_sp_ctx* c, const double* source_host) {
    if (!c) return LBM_EINVAL;
    if (!source_host) return sp_fail(c, LBM_EINVAL, "source is NULL");
    cudaError_t r;
    if ((r = cudaMemcpyAsync(c->d_tmp, source_host, c->N * sizeof(double), cudaMemcpyHostToDevice,
                             c->stream)) != cudaSuccess)
        return sp_cuda(c, r, "source upload");
    if (c->form == LBM_F64) {
        sp_convert_kernel<double><<<blocks(c->N), 256, 0, c->stream>>>(c->d_tmp, static_cast<double*>(c->src), c->N);
    } else {
        sp_convert_kernel<float><<<blocks(c->N), 256, 0, c->stream>>>(c->d_tmp, static_cast<float*>(c->src), c->N);
    }
    c->cur = 0;
    // at rest: Remark 3 g^eq = rho_0 delta_i0 (g_0 stored shifted by rho_0);
    // Remark 1 g^eq = w_i at rho = 1, Remark 2 w_i p_0 (stored shifted by
    // them) -- zero in every case
    if ((r = cudaMemsetAsync(c->g[0], 0, kQ * c->N * sp_elem(c->form), c->stream)) != cudaSuccess)
        return sp_cuda(c, r, "state reset");
    // Remark 4 scheme: u at t = -1 is u at t = 0 = 0
    if (c->p.scheme == LBM_SP_SCHEME_REMARK4 &&
        (r = cudaMemsetAsync(c->ufield, 0, 2 * c->N * sp_elem(c->form), c->stream)) != cudaSuccess)
        return sp_cuda(c, r, "state reset");
    if ((r = cudaMemsetAsync(c->d_status, 0, sizeof(int), c->stream)) != cudaSuccess) return sp_cuda(c, r, "state reset");
    if ((r = cudaStreamSynchronize(c->stream)) != cudaSuccess) return sp_cuda(c, r, "init");
    if ((r = cudaGetLastError()) != cudaSuccess) return sp_cuda(c, r, "init kernel");
    c->ready = true;
    c->time = 0;
    return LBM_OK;
}

lbm_status lbm_sp_step(lbm_sp_ctx* c, int nsteps) {
    if (!c) return LBM_EINVAL;
    if (nsteps < 0) return sp_fail(c, LBM_EINVAL, "nsteps < 0");
    if (!c->ready) return sp_fail(c, LBM_ESTATE, "not initialised");
    for (int s = 0; s < nsteps;) {
        const int n = c->tile ? (nsteps - s < 256 ? nsteps - s : 256) : 1;
        const cudaError_t e = c->tile ? sp_step_tiles(c, n) : sp_step_once(c);
        if (e != cudaSuccess) return sp_cuda(c, e, "step kernel");
        s += n;
    }
    c->time += nsteps;
    const cudaError_t r = cudaGetLastError();
    return r == cudaSuccess ? LBM_OK : sp_cuda(c, r, "step kernel");
}

lbm_status lbm_sp_get_fields(lbm_sp_ctx* c, unsigned mask, double* host_out) {
    if (!c) return LBM_EINVAL;
    const bool m1 = c->p.model == LBM_SP_NEARLY_INCOMPRESSIBLE, m2 = c->p.model == LBM_SP_HE_INCOMPRESSIBLE;
    const unsigned ok = LBM_FIELD_UX | LBM_FIELD_UY | LBM_FIELD_P | (m1 ? LBM_FIELD_RHO : 0u);
    if (!host_out || mask == 0 || (mask & ~ok)) return sp_fail(c, LBM_EINVAL, "bad mask or output");
    if (!c->ready) return sp_fail(c, LBM_ESTATE, "not initialised");
    const int nf = ((mask & LBM_FIELD_UX) ? 1 : 0) + ((mask & LBM_FIELD_UY) ? 1 : 0) + ((mask & LBM_FIELD_P) ? 1 : 0) +
                   ((mask & LBM_FIELD_RHO) ? 1 : 0);
    if (c->p.scheme == LBM_SP_SCHEME_REMARK4 && c->form == LBM_F64)
        sp4_fields_kernel<double><<<blocks(c->N), 256, 0, c->stream>>>(
            static_cast<const double*>(c->g[c->cur]), static_cast<const double*>(c->src), c->N, c->K, mask, c->d_tmp);
    else if (c->p.scheme == LBM_SP_SCHEME_REMARK4)
        sp4_fields_kernel<float><<<blocks(c->N), 256, 0, c->stream>>>(
            static_cast<const float*>(c->g[c->cur]), static_cast<const float*>(c->src), c->N, c->K, mask, c->d_tmp);
    else if (m1)
        sp1_fields<1>(c, mask);
    else if (m2)
        sp1_fields<2>(c, mask);
    else if (c->form == LBM_F64)
        sp_fields_kernel<double><<<blocks(c->N), 256, 0, c->stream>>>(
            static_cast<const double*>(c->g[c->cur]), static_cast<const double*>(c->src), c->N, c->K, mask, c->d_tmp);
    else
        sp_fields_kernel<float><<<blocks(c->N), 256, 0, c->stream>>>(
            static_cast<const float*>(c->g[c->cur]), static_cast<const float*>(c->src), c->N, c->K, mask, c->d_tmp);
    cudaError_t r;
    if ((r = cudaMemcpyAsync(host_out, c->d_tmp, nf * c->N * sizeof(double), cudaMemcpyDeviceToHost,
                             c->stream)) != cudaSuccess)
        return sp_cuda(c, r, "fields read-back");
    if ((r = cudaStreamSynchronize(c->stream)) != cudaSuccess) return sp_cuda(c, r, "fields");
    return sp_device_status(c);
}

lbm_status lbm_sp_get_populations(lbm_sp_ctx* c, double* host_g) {
    if (!c) return LBM_EINVAL;
    if (!host_g) return sp_fail(c, LBM_EINVAL, "output is NULL");
    if (!c->ready) return sp_fail(c, LBM_ESTATE, "not initialised");
    const long long n = kQ * c->N;
    const bool shifted = c->p.model == LBM_SP_NEARLY_INCOMPRESSIBLE || c->p.model == LBM_SP_HE_INCOMPRESSIBLE;
    const double a0 = c->p.model == LBM_SP_HE_INCOMPRESSIBLE ? c->p.p0 : 1.0;   // the stored shift w_i a0
    if (shifted && c->form == LBM_F64)
        sp1_widen_kernel<double><<<blocks(c->N), 256, 0, c->stream>>>(static_cast<const double*>(c->g[c->cur]),
                                                                      c->d_tmp, c->N, a0);
    else if (shifted)
        sp1_widen_kernel<float><<<blocks(c->N), 256, 0, c->stream>>>(static_cast<const float*>(c->g[c->cur]),
                                                                     c->d_tmp, c->N, a0);
    else if (c->form == LBM_F64)
        sp_widen_kernel<double><<<blocks(n), 256, 0, c->stream>>>(static_cast<const double*>(c->g[c->cur]), c->d_tmp, n);
    else
        sp_widen_kernel<float><<<blocks(n), 256, 0, c->stream>>>(static_cast<const float*>(c->g[c->cur]), c->d_tmp, n);
    cudaError_t r;
    if ((r = cudaMemcpyAsync(host_g, c->d_tmp, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream)) != cudaSuccess)
        return sp_cuda(c, r, "populations read-back");
    if ((r = cudaStreamSynchronize(c->stream)) != cudaSuccess) return sp_cuda(c, r, "populations");
    return sp_device_status(c);
}

const char* lbm_sp_last_error(const lbm_sp_ctx* c) { return c ? c->err.c_str() : "null context"; }

void lbm_sp_destroy(lbm_sp_ctx* c) {
    if (!c) return;
    sp_release(c);
    delete c;
}

}  // extern "C"
