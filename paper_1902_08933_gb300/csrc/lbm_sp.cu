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
#include "lbm_device.cuh"

namespace {

constexpr int kQ = 9;
__host__ __device__ constexpr int sx(int i) { return i == 1 || i == 5 || i == 8 ? 1 : (i == 3 || i == 6 || i == 7 ? -1 : 0); }
__host__ __device__ constexpr int sy(int i) { return i == 2 || i == 5 || i == 6 ? 1 : (i == 4 || i == 7 || i == 8 ? -1 : 0); }
__host__ __device__ constexpr double sw(int i) { return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0); }
__host__ __device__ constexpr int sopp(int i) { return i == 0 ? 0 : (i <= 4 ? (i + 1) % 4 + 1 : (i - 5 + 2) % 4 + 5); }
static_assert(sopp(1) == 3 && sopp(2) == 4 && sopp(5) == 7 && sopp(6) == 8 && sopp(8) == 6, "D2Q9 opposites");
// one direction of each opposite pair (1, 2, 5, 6; their opposites 3, 4, 7, 8)
__host__ __device__ constexpr int pair2(int q) { return q == 0 ? 1 : q == 1 ? 2 : q == 2 ? 5 : 6; }

// ---- Arithmetic ----
// A unit of the step: one cell (One<float>, One<double>), or two horizontally
// adjacent ones (x, x + 1), x even, in packed FP32 instructions (Two; nx even). No
// sum below is left to the compiler to contract: a velocity component that the flow
// does not have (u_y of a source that does not vary in y) is nothing but the rounding
// residue of these sums, so which products are rounded before they are added is part
// of the results, and the same in every kernel. For the packed instructions, which
// the compiler contracts where it likes, that takes additions as FFMA2 with a factor
// that it cannot know to be 1 or -1.
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
template <typename T> __device__ __forceinline__ One<T> operator-(One<T> a) { return One<T>(-a.v); }

__constant__ float2 sp_plus = {1.f, 1.f}, sp_minus = {-1.f, -1.f};   // (never written)
struct Two {
    float2 v;
    Two() = default;
    __device__ __forceinline__ Two(float s) : v(make_float2(s, s)) {}
    __device__ __forceinline__ Two(float a, float b) : v(make_float2(a, b)) {}
    __device__ __forceinline__ explicit Two(float2 w) : v(w) {}
};
__device__ __forceinline__ Two operator+(Two a, Two b) { return Two(__ffma2_rn(b.v, sp_plus, a.v)); }
__device__ __forceinline__ Two operator-(Two a, Two b) { return Two(__ffma2_rn(b.v, sp_minus, a.v)); }
__device__ __forceinline__ Two operator*(Two a, Two b) { return Two(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ Two operator-(Two a) { return Two(-a.v.x, -a.v.y); }
__device__ __forceinline__ Two fmadd(Two a, Two b, Two c) { return Two(__ffma2_rn(a.v, b.v, c.v)); }

// c + a b and c - a b, rounded once by a single cell, the product first by a pair
template <typename T>
__device__ __forceinline__ One<T> add_prod(One<T> c, One<T> a, One<T> b) { return fmadd(a, b, c); }
template <typename T>
__device__ __forceinline__ One<T> sub_prod(One<T> c, One<T> a, One<T> b) { return fmadd(-a, b, c); }
__device__ __forceinline__ Two add_prod(Two c, Two a, Two b) { return c + a * b; }
__device__ __forceinline__ Two sub_prod(Two c, Two a, Two b) { return c - a * b; }
// a b - c d: the first product not rounded by a single cell, both rounded by a pair
template <typename T>
__device__ __forceinline__ One<T> diff_prod(One<T> a, One<T> b, One<T> c, One<T> d) { return fmadd(a, b, -(c * d)); }
__device__ __forceinline__ Two diff_prod(Two a, Two b, Two c, Two d) { return a * b - c * d; }
// 1/x and sqrt(x), correctly rounded per cell
template <typename T> __device__ __forceinline__ One<T> sp_inv(One<T> x) { return One<T>(T(1) / x.v); }
template <typename T> __device__ __forceinline__ One<T> sp_sqrt(One<T> x) { return One<T>(sqrt(x.v)); }
__device__ __forceinline__ Two sp_inv(Two x) { return Two(1.f / x.v.x, 1.f / x.v.y); }
__device__ __forceinline__ Two sp_sqrt(Two x) { return Two(sqrtf(x.v.x), sqrtf(x.v.y)); }

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
template <> struct Unit<Two> {
    using R = float;
    using E = float2;
    static constexpr int cells = 2;
    __device__ __forceinline__ static Two ld(const float* p) { return Two(*reinterpret_cast<const float2*>(p)); }
    __device__ __forceinline__ static void st(float* p, Two v) { *reinterpret_cast<float2*>(p) = v.v; }
    __device__ __forceinline__ static E pack(Two v) { return v.v; }
    __device__ __forceinline__ static Two at(const E* row, int t, int dx) {
        if (dx < 0) return Two(row[t - 1].y, row[t].x);
        if (dx > 0) return Two(row[t].y, row[t + 1].x);
        return Two(row[t]);
    }
    __device__ __forceinline__ static void push(float* row, int x, int nx, int dx, Two v) {
        if (dx == 0) {   // keeps the pair together
            st(row + x, v);
        } else {
            row[dx < 0 ? (x == 0 ? nx - 1 : x - 1) : x + 1] = v.v.x;
            row[dx < 0 ? x : (x + 2 == nx ? 0 : x + 2)] = v.v.y;
        }
    }
};

// Constants of a model: FP64, and for FP32 contexts converted on the host, so that
// their kernels do no FP64 arithmetic.
template <typename T>
struct SpConst {
    int nx, ny, walls;
    T inv_tau, src, tgm, Qc, fx, fy;   // 1/tau_g, 1 - 1/(2 tau_g), tau_g - 1/2, Q, F
    T dl, dq;                          // drag of the Remark 4 scheme: F(u) = F - (dl + dq |u|) u
    T p0;                              // Remark 2: the constant p_0
    T tau, Qd0;                        // tau_g; Q - (2/d) c_s^2 (the part of Q without the density)
    T hp0, ip0, hp0fx, hp0fy;          // p_0 / 2, 1 / p_0, p_0 F_1 / 2
};
template <typename T>
SpConst<T> sp_const_as(const SpConst<double>& K) {
    return SpConst<T>{K.nx, K.ny, K.walls, T(K.inv_tau), T(K.src), T(K.tgm), T(K.Qc), T(K.fx), T(K.fy),
                      T(K.dl), T(K.dq), T(K.p0), T(K.tau), T(K.Qd0), T(K.hp0), T(K.ip0), T(K.hp0fx), T(K.hp0fy)};
}
// 4.5 (|c_i|^2 - 2/3), rounded in the arithmetic type
template <typename T>
__device__ __forceinline__ constexpr T sp_c2(int i) {
    return T(4.5) * (T(sx(i) * sx(i) + sy(i) * sy(i)) - T(2.0 / 3.0));
}

// ---- Moments, of the step and of the read-back: the u handed out is the u the step
// collides with ----
// sum c_i g_i, one population after the other
template <typename V>
__device__ __forceinline__ void sp_j(const V (&g)[kQ], V& jx, V& jy) {
    jx = g[1];
    jy = g[2];
#pragma unroll
    for (int i = 3; i < kQ; ++i) {
        if (sx(i)) jx = sx(i) > 0 ? jx + g[i] : jx - g[i];
        if (sy(i)) jy = sy(i) > 0 ? jy + g[i] : jy - g[i];
    }
}
template <typename V>
__device__ __forceinline__ V sp_rest(const V (&g)[kQ]) {
    V s = g[1];
#pragma unroll
    for (int i = 2; i < kQ; ++i) s = s + g[i];
    return s;
}

// Remark 3: u (Eq. 27a, rho = 1), u.F, u.u, G_0 and p (Eq. 28)
template <typename V>
struct SpCell { V ux, uy, uF, uu, G0, p; };
template <typename V, typename T>
__device__ __forceinline__ SpCell<V> sp3_moments(const SpConst<T>& K, const V (&g)[kQ], V S) {
    SpCell<V> m;
    V jx, jy;
    sp_j(g, jx, jy);
    m.ux = jx + V(T(0.5) * K.fx);
    m.uy = jy + V(T(0.5) * K.fy);
    m.uF = fmadd(m.ux, V(K.fx), m.uy * V(K.fy));
    m.uu = fmadd(m.ux, m.ux, m.uy * m.uy);
    m.G0 = V(T(sw(0))) * fmadd(V(sp_c2<T>(0)), V(K.Qc) * S, sub_prod(S, V(T(3)), m.uF));
    // c_s^2 / (1 - w_0) = 3/5; s_0(u) = -w_0 u.u / (2 c_s^2) = -(2/3) u.u
    m.p = V(T(0.6)) * fmadd(V(K.tgm), m.G0, sub_prod(sp_rest(g) + V(T(0.5)) * S, V(T(2.0 / 3.0)), m.uu));
    return m;
}

// Remarks 1 and 2 (M = 1, 2): g holds g_i - w_i a0 (a0 = 1 for Remark 1, p_0 for
// Remark 2: the rest state). d = rho - 1 (Remark 1) or p - p_0 (Remark 2); a = rho or
// p_0, the factor of s_i(u) in g^eq (Eq. 29bb, Eq. 29bd); both equilibria are d w_i +
// a s_i(u) after the shift.
template <int M, typename V, typename T>
__device__ __forceinline__ void sp1_moments(const SpConst<T>& K, const V (&g)[kQ], V S, V& d, V& a, V& ux, V& uy) {
    V m0 = g[0], jx, jy;
    sp_j(g, jx, jy);
#pragma unroll
    for (int i = 1; i < kQ; ++i) m0 = m0 + g[i];
    if constexpr (M == 1) {
        d = m0 + V(T(0.5)) * S;                       // Eq. 27aa
        a = V(T(1)) + d;
        const V ir = sp_inv(a);
        ux = (jx + V(T(0.5) * K.fx)) * ir;            // Eq. 27a
        uy = (jy + V(T(0.5) * K.fy)) * ir;
    } else {
        d = fmadd(V(K.hp0), S, m0);                   // p = sum g + p_0 S_1 / 2
        a = V(K.p0);
        ux = (jx + V(K.hp0fx)) * V(K.ip0);            // p_0 u = sum c g + p_0 F_1 / 2
        uy = (jy + V(K.hp0fy)) * V(K.ip0);
    }
}

// Remark 4 scheme: F(u)
template <typename V, typename T>
__device__ __forceinline__ void sp4_force(const SpConst<T>& K, V ux, V uy, V& Fx, V& Fy) {
    const V k = fmadd(V(K.dq), sp_sqrt(fmadd(ux, ux, uy * uy)), V(K.dl));
    Fx = sub_prod(V(K.fx), k, ux);
    Fy = sub_prod(V(K.fy), k, uy);
}
// G_0 / w_0
template <typename V, typename T>
__device__ __forceinline__ V sp4_G0w(const SpConst<T>& K, V S, V uF) {
    return fmadd(V(sp_c2<T>(0) * K.Qc), S, sub_prod(S, V(T(3)), uF));
}
// p (Eq. 28 for the unshifted f, tau_g G_0)
template <typename V, typename T>
__device__ __forceinline__ V sp4_p(const SpConst<T>& K, const V (&f)[kQ], V uu, V G0) {
    return V(T(0.6)) * fmadd(V(K.tau), G0, sub_prod(sp_rest(f), V(T(2.0 / 3.0)), uu));
}

// ---- Read-back ----
template <int M, typename R>
__global__ void sp1_fields_kernel(const R* __restrict__ g, const R* __restrict__ src, long long N, SpConst<R> K,
                                  double p0, unsigned mask, double* __restrict__ out) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    One<R> gc[kQ], d, a, ux, uy;
#pragma unroll
    for (int i = 0; i < kQ; ++i) gc[i] = g[i * N + c];
    sp1_moments<M>(K, gc, One<R>(src[c]), d, a, ux, uy);
    // Remark 1: p = rho c_s^2, rho = 1 + d; Remark 2: p = p_0 + d
    const double p = M == 1 ? (1.0 + double(d.v)) / 3.0 : p0 + double(d.v);
    int slot = 0;
    if (mask & LBM_FIELD_UX) out[(slot++) * N + c] = double(ux.v);
    if (mask & LBM_FIELD_UY) out[(slot++) * N + c] = double(uy.v);
    if (mask & LBM_FIELD_P) out[(slot++) * N + c] = p;
    if (M == 1 && (mask & LBM_FIELD_RHO)) out[(slot++) * N + c] = 1.0 + double(d.v);
}

// Remark 3, or (R4) the Remark 4 scheme
template <bool R4, typename R>
__global__ void sp_fields_kernel(const R* __restrict__ g, const R* __restrict__ src, long long N, SpConst<R> K,
                                 unsigned mask, double* __restrict__ out) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    One<R> gc[kQ], ux, uy, p;
#pragma unroll
    for (int i = 0; i < kQ; ++i) gc[i] = g[i * N + c];
    const One<R> S(src[c]);
    if constexpr (R4) {
        One<R> Fx, Fy;
        sp_j(gc, ux, uy);
        sp4_force(K, ux, uy, Fx, Fy);
        const One<R> G0 = One<R>(R(sw(0))) * sp4_G0w(K, S, fmadd(ux, Fx, uy * Fy));
        p = sp4_p(K, gc, fmadd(ux, ux, uy * uy), G0);
    } else {
        const SpCell<One<R>> m = sp3_moments(K, gc, S);
        ux = m.ux;
        uy = m.uy;
        p = m.p;
    }
    int slot = 0;
    if (mask & LBM_FIELD_UX) out[(slot++) * N + c] = double(ux.v);
    if (mask & LBM_FIELD_UY) out[(slot++) * N + c] = double(uy.v);
    if (mask & LBM_FIELD_P) out[(slot++) * N + c] = double(p.v);
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
// The four models by one number: Remarks 1, 2, 3 and the Remark 4 scheme.
// What a cell's neighbours need of it (values of the shared-memory ring): u for
// div u (Remarks 1, 2), G_i / w_i, i = 1 .. 8, for G_i at x + c_i (Remark 4),
// nothing (3).
template <int KIND> constexpr int kRing = KIND == 4 ? 8 : (KIND == 3 ? 0 : 2);

// A cell's own values besides its populations and S.
template <typename V>
struct SpMom { V ux, uy, a, b; };   // u; Remarks 1, 2: d and a of the equilibrium; Remark 4: F(u)

// c_i.(x, y) of the directions 1, 2, 5, 6
template <typename V>
__device__ __forceinline__ V sp_dot(int i, V x, V y) { return i == 1 ? x : i == 2 ? y : i == 5 ? x + y : y - x; }

// u and what the neighbours need (put(r, value): ring value r).
template <int KIND, typename V, typename T, typename Put>
__device__ __forceinline__ void sp_moments_of(const SpConst<T>& K, const V (&g)[kQ], V S, SpMom<V>& m, Put&& put) {
    if constexpr (KIND == 4) {
        sp_j(g, m.ux, m.uy);   // u = sum c f
        sp4_force(K, m.ux, m.uy, m.a, m.b);
        const V uF = fmadd(m.ux, m.a, m.uy * m.b), three(T(3));
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = pair2(q);
            const V cu9 = V(T(9)) * sp_dot(i, m.ux, m.uy), cF = sp_dot(i, m.a, m.b), cQ(sp_c2<T>(i) * K.Qc);
            put(i - 1, fmadd(cQ, S, sub_prod(fmadd(cu9, cF, fmadd(three, cF, S)), three, uF)));
            put(sopp(i) - 1, fmadd(cQ, S, sub_prod(fmadd(cu9, cF, fmadd(-three, cF, S)), three, uF)));
        }
    } else if constexpr (KIND != 3) {
        sp1_moments<KIND>(K, g, S, m.a, m.b, m.ux, m.uy);
        put(0, m.ux);
        put(1, m.uy);
    }
}

// Remark 4: the parts of G_i even in c and of c_i.F / c_s^2 (o, without w_i) at velocity u
template <typename V, typename T>
__device__ __forceinline__ void sp4_parts(const SpConst<T>& K, int i, V S, V ux, V uy, V Fx, V Fy, V uF, V& e, V& o) {
    const V cF = sp_dot(i, Fx, Fy), cQ(sp_c2<T>(i) * K.Qc);
    const V b = sub_prod(fmadd(V(T(9)) * sp_dot(i, ux, uy), cF, S), V(T(3)), uF);
    e = V(T(sw(i))) * (i >= 5 ? b + cQ * S : fmadd(cQ, S, b));
    o = V(T(3)) * cF;
}

// Collision (Eq. 24 with the remark's equilibrium and force term) in opposite pairs of
// directions: the parts of s_i and G_i even in c shared, the odd parts flipped.
// nb(r, dx, dy): ring value r of a neighbour (mirrored about a wall); up: u at t - 1
// (Remark 4); emit(i, value, wall): the population leaving in direction i, and a
// function giving what returns if a wall reflects it (the same but for Remark 4).
// (c c - c_s^2 I):(u F + F u [- u u S] + Q D I) / (2 c_s^4) = 9 (c.u)(c.F) - 3 u.F
// [- 4.5 ((c.u)^2 - u.u / 3) S] + 4.5 (|c|^2 - 2/3) Q D; D = S, or div u (Remarks 1, 2).
template <int KIND, typename V, typename T, typename Nb, typename Emit>
__device__ __forceinline__ void sp_collide(const SpConst<T>& K, const V (&g)[kQ], V S, const SpMom<V>& m, V upx, V upy,
                                           Nb&& nb, Emit&& emit) {
    constexpr bool pair = Unit<V>::cells == 2;
    constexpr T w0d = T(sw(0)), w01 = pair ? T(sw(0) - 1.0) : w0d - T(1);   // w_0, w_0 - 1
    const V w0(w0d), ig(K.inv_tau), sg(K.src), three(T(3)), half(T(0.5));
    auto relax = [&](V gi, V geq) { return sub_prod(gi, gi - geq, ig); };
    if constexpr (KIND == 3) {
        const SpCell<V> c = sp3_moments(K, g, S);
        const V QS = V(K.Qc) * S, p3 = three * c.p;
        const V r0 = fmadd(sg, c.G0, relax(g[0], fmadd(p3, V(w01), w0 * (V(T(-1.5)) * c.uu))));
        emit(0, r0, [&] { return r0; });
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = pair2(q), j = sopp(i);
            const V w(T(sw(i))), cu = sp_dot(i, c.ux, c.uy), cF = sp_dot(i, V(K.fx), V(K.fy)), y = three * cF;
            const V e = w * fmadd(V(sp_c2<T>(i)), QS, sub_prod(fmadd(V(T(9)) * cu, cF, S), three, c.uF));
            const V cu2 = V(T(4.5)) * cu * cu, pw = p3 * w;
            const V si = sub_prod(fmadd(three, cu, cu2), V(T(1.5)), c.uu);
            const V sj = sub_prod(fmadd(-three, cu, cu2), V(T(1.5)), c.uu);
            const V ri = fmadd(sg, add_prod(e, w, y), relax(g[i], fmadd(w, si, pw)));
            const V rj = fmadd(sg, sub_prod(e, w, y), relax(g[j], fmadd(w, sj, pw)));
            emit(i, ri, [&] { return ri; });
            emit(j, rj, [&] { return rj; });
        }
    } else if constexpr (KIND == 4) {
        const V ux = m.ux, uy = m.uy, Fx = m.a, Fy = m.b;
        const V uu = fmadd(ux, ux, uy * uy), uF = fmadd(ux, Fx, uy * Fy);
        const V G0 = w0 * sp4_G0w(K, S, uF), p = sp4_p(K, g, uu, G0), p3 = three * p;
        V Fpx, Fpy;   // F at t - 1
        sp4_force(K, upx, upy, Fpx, Fpy);
        const V upF = fmadd(upx, Fpx, upy * Fpy);
        {   // rest direction: its destination is this cell
            const V z = V(T(-1.5)) * uu;
            V geq;
            if constexpr (pair) geq = fmadd(p3, V(w01), w0 * z);
            else geq = fmadd(w0, z, p3 * V(w01));
            emit(0, fmadd(half, sub_prod(G0, w0, sp4_G0w(K, S, upF)), relax(g[0], geq) + G0), [] { return V(T(0)); });
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = pair2(q), j = sopp(i);
            const V w(T(sw(i))), cu = sp_dot(i, ux, uy);
            const V E = diff_prod(V(T(4.5)) * cu, cu, V(T(1.5)), uu);
            V ge;
            if constexpr (pair) ge = fmadd(w, E, V(T(3) * T(sw(i))) * p);
            else ge = i >= 5 ? fmadd(w, E, p3 * w) : fmadd(p3, w, w * E);
            V Ge, Gy, Pe, Py;
            sp4_parts(K, i, S, ux, uy, Fx, Fy, uF, Ge, Gy);
            sp4_parts(K, i, S, upx, upy, Fpx, Fpy, upF, Pe, Py);
            const V Gi = add_prod(Ge, w, Gy), Gj = sub_prod(Ge, w, Gy);
            const V Pi = add_prod(Pe, w, Py), Pj = sub_prod(Pe, w, Py);
            const V xi = nb(i - 1, sx(i), sy(i)), xj = nb(j - 1, sx(j), sy(j));   // G / w at the destinations
            // G_i(x + c_i, t) - G_i(x, t - 1)
            auto change = [&](V x, V P) { return !pair && sy(i) == 0 ? fmadd(w, x, -P) : w * x - P; };
            const V cy = three * cu;
            const V pi = fmadd(half, change(xi, Pi), relax(g[i], add_prod(ge, w, cy)) + Gi);
            const V pj = fmadd(half, change(xj, Pj), relax(g[j], sub_prod(ge, w, cy)) + Gj);
            // bounce-back of f - G/2: leaves as i with G_i(x + c_i), returns as opp(i)
            emit(i, pi, [&] { return fmadd(half, Gj, fmadd(-half, w * xi, pi)); });
            emit(j, pj, [&] { return fmadd(half, Gi, fmadd(-half, w * xj, pj)); });
        }
    } else {
        const V ux = m.ux, uy = m.uy, d = m.a, a = m.b;
        V divu(T(0));   // Eq. 30a applied to u; pairs sum row by row
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            constexpr int by_row[8] = {4, 7, 8, 1, 3, 2, 5, 6};
            const int i = pair ? by_row[k] : k + 1;
            V cu;
            if (sy(i) == 0) cu = nb(0, sx(i), 0);
            else if (sx(i) == 0) cu = nb(1, 0, sy(i));
            else cu = sx(i) * sy(i) > 0 ? nb(0, sx(i), sy(i)) + nb(1, sx(i), sy(i)) : nb(0, sx(i), sy(i)) - nb(1, sx(i), sy(i));
            // (a sign for the direction as a whole)
            divu = fmadd(V((sx(i) ? sx(i) : sy(i)) * T(sw(i))), cu, divu);
        }
        divu = divu * three;
        const V third(T(1.0 / 3.0));
        const V Qd = fmadd(a, third, V(K.Qd0)) * divu;   // Q div u, Q = (2/d) a c_s^2 - xi / (tau_g - 1/2)
        // S and F in the units of g
        const V fx(KIND == 1 ? K.fx : K.fx * K.p0), fy(KIND == 1 ? K.fy : K.fy * K.p0);
        V Sg = S;
        if constexpr (KIND == 2) Sg = S * V(K.p0);
        const V uF = fmadd(ux, fx, uy * fy), uu = fmadd(ux, ux, uy * uy);
        auto source = [&](V G, V cc) {   // the u u S of Remark 1: cc = (c.u)^2 - u.u / 3
            if constexpr (KIND == 1) return sub_prod(G, V(T(4.5)) * cc, Sg);
            else return G;
        };
        {
            const V geq = fmadd(d, w0, a * (w0 * (V(T(-1.5)) * uu)));
            const V G = source(fmadd(V(sp_c2<T>(0)), Qd, sub_prod(Sg, three, uF)), -(uu * third));
            const V r0 = fmadd(sg, w0 * G, relax(g[0], geq));
            emit(0, r0, [&] { return r0; });
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = pair2(q), j = sopp(i);
            const bool diag = i >= 5;
            const V w(T(sw(i))), cu = sp_dot(i, ux, uy), cF = sp_dot(i, fx, fy), c2(sp_c2<T>(i));
            const V wE = w * diff_prod(V(T(4.5)) * cu, cu, V(T(1.5)), uu);
            const V ge = pair || diag ? fmadd(a, wE, d * w) : fmadd(d, w, a * wE), o = w * (three * cu);
            V G = sub_prod(fmadd(V(T(9)) * cu, cF, Sg), three, uF);
            G = pair && diag ? G + c2 * Qd : fmadd(c2, Qd, G);
            if constexpr (KIND == 1) G = source(G, diff_prod(cu, cu, uu, third));
            const V e = w * G, y = three * cF;
            const V ri = fmadd(sg, add_prod(e, w, y), relax(g[i], add_prod(ge, a, o)));
            const V rj = fmadd(sg, sub_prod(e, w, y), relax(g[j], sub_prod(ge, a, o)));
            emit(i, ri, [&] { return ri; });
            emit(j, rj, [&] { return rj; });
        }
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
    __device__ __forceinline__ SpPush(const SpConst<T>& K, typename U::R* out_, int N_, int x_, int y_)
        : out(out_), N(N_), nx(K.nx), x(x_), y(y_) {
        bot = K.walls && y == 0;
        top = K.walls && y == K.ny - 1;
        dn = y == 0 ? K.ny - 1 : y - 1;   // (not used at a wall)
        up = y == K.ny - 1 ? 0 : y + 1;
    }
    template <typename Wall>
    __device__ __forceinline__ void operator()(int i, V v, Wall&& wall) const {
        if ((sy(i) > 0 && top) || (sy(i) < 0 && bot)) {
            U::st(out + sopp(i) * N + y * nx + x, wall());
            return;
        }
        U::push(out + i * N + (sy(i) == 0 ? y : (sy(i) > 0 ? up : dn)) * nx, x, nx, sx(i), v);
    }
};

// Remark 3, large domains: nothing of a neighbour is needed, one unit a thread.
// 4096 x 4096 FP32 188 us a step (1.0 of the copy bandwidth); FP64 bound by its FP64
// operations, 2048 x 2048 1076 us.
template <typename V>
__global__ void __launch_bounds__(256, sizeof(typename Unit<V>::R) == 8 ? 3 : 4)
    sp_cell_kernel(const typename Unit<V>::R* __restrict__ gin, typename Unit<V>::R* __restrict__ gout,
                   const typename Unit<V>::R* __restrict__ src, int N, SpConst<typename Unit<V>::R> K) {
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
// 4096 x 4096 FP32, two kernels -> here, us a step: Remark 1 375 -> 232 (0.81 of
// the copy bandwidth), 2 330 -> 223 (0.85), 4 489 -> 322 (0.71: three quarters of it
// arithmetic at 16 warps a SM); 2048 x 2048 FP64 (bound by its FP64 operations either
// way: the moments are formed once instead of twice) 1790 -> 1369, 1525 -> 1198, 2459 ->
// 2227. Bit for bit the two kernels' results (see "Arithmetic").
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
    __device__ __forceinline__ SpMarch(const SpConst<T>& K, const SpRun& r) : ny(K.ny), walls(K.walls) {
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
                                                                   SpConst<typename Unit<V>::R> K, SpRun run) {
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
    int N, nitems, nsteps, ulog, wait_limit, wait_extra;   // wait_*: as in StepArgs
    const lbm::WorkItem* work;
    const int* nbr;
    int *done, *status;
};

template <int KIND, typename V, int OCC>
__global__ void __launch_bounds__(kSpThreads, OCC) sp_tile_kernel(const SpTileArgs a, SpConst<typename Unit<V>::R> K) {
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
            if (s > 0 && !lbm::tile_wait(a.done, a.nbr + item * lbm::kMaxTileNbr, s + a.wait_extra, a.wait_limit,
                                         a.status, a.done + a.nitems, &s_bad, tid))
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
    SpConst<double> K{};
    SpConst<float> kf{};               // FP32 steps: the constants in FP32
    int kind = 3;                      // 1, 2, 3: Remarks; 4: the Remark 4 scheme
    int cells = 1;                     // cells a unit: 2 in FP32 with nx even
    const void* kernel = nullptr;      // one step a launch: row march, Remark 3 one unit a thread
    SpRun run{};
    int threads = kSpThreads;
    const void* tile = nullptr;        // small domains: several steps a launch (null: not taken)
    int tile_items = 0, tile_grid = 0, tile_ulog = 0;
    lbm::ItemBuffers tile_buf;         // items, neighbours, step counters and abort flag
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
    c->tile_buf.release();
    cudaFree(c->d_status);
    cudaFree(c->d_tmp);
    if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
}

// The step kernels of a model for unit type V, and the resident blocks of 128
// threads a SM their registers are sized for. The row march holds two rows of
// populations and a third in flight. us a step of the marches with 3 / 4 / 5 blocks:
// pairs (4096 x 4096) Remark 1 256 / 232 / 287, Remark 2 244 / 223 / 227, Remark 4 357 /
// 322 / 461; one FP32 cell (4095 x 4096) with 4 / 5 / 6 blocks 287 / 268 / 283, 275 / 257 /
// 255, 422 / 372 / 435; FP64 (2048 x 2048) with 2 / 3 / 4: 1369 / 1401 / 1488, 1198 / 1232 /
// 1314, 2306 / 2227 / 2361. Tiles: FP64 with 3 and 5 blocks 256 x 256 39.7 and 27.8, 34.1
// and 23.9, 66.2 and 45.9 (one round of tiles for two), 192 x 192 (one either way) the same.
template <typename V>
void sp_kernels(int kind, const void** step, const void** tile) {
    constexpr bool f64 = sizeof(typename Unit<V>::R) == 8, pair = Unit<V>::cells == 2;
    constexpr int m = f64 ? 2 : pair ? 4 : 5, m4 = f64 ? 3 : pair ? 4 : 5;
    constexpr int o = f64 ? 5 : pair ? 4 : 6;
    switch (kind) {
        case 1:
            *step = (const void*)sp_march_kernel<1, V, m>;
            *tile = (const void*)sp_tile_kernel<1, V, o>;
            break;
        case 2:
            *step = (const void*)sp_march_kernel<2, V, m>;
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
    c->kf = sp_const_as<float>(c->K);
    c->cells = c->form == LBM_F32 && c->p.nx % 2 == 0 ? 2 : 1;
    if (c->form == LBM_F64) sp_kernels<One<double>>(c->kind, &c->kernel, &c->tile);
    else if (c->cells == 2) sp_kernels<Two>(c->kind, &c->kernel, &c->tile);
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
            lbm::each_run_length(c->p.ny, [&](int rows) {
                const int runs = (c->p.ny + rows - 1) / rows;
                const long long cost = ((long long)strips * runs + target - 1) / target * (rows + 2);
                if (best < 0 || cost < best) {
                    best = cost;
                    c->threads = threads;
                    c->run = SpRun{rows, strips, w * c->cells};
                }
                return true;
            });
        }
    }
    // Tiles, several steps a launch, while every tile is resident at once: a step of
    // a small domain is the latency of a launch. us a step, tiles and one launch a
    // step: 64 x 64 Remark 1 FP32 3.0 and 4.1, FP64 7.7 and 12.3; 256 x 256 3.8 and 6.2,
    // 27.8 and 41.0; 300 x 300 4.1 and 6.2, 35.8 and 41.0; in two rounds 400 x 400 FP32
    // 8.8 and 8.2, 340 x 340 FP64 60 and 57.
    auto count = [&](int u, int r) { return (long long)((units + u - 1) / u) * ((c->p.ny + r - 1) / r); };
    int U, R;
    lbm::tile_shape(count, sms, &U, &R);
    const long long tslots = slots(c->tile, kSpThreads);
    if (count(8, 16) < count(U, R) && count(U, R) > tslots) {
        U = 8;
        R = 16;
    }
    if (count(U, R) > tslots) {
        c->tile = nullptr;
        return LBM_OK;
    }
    lbm::TileList list;
    lbm::add_tiles(list, 0, c->p.nx, c->p.ny, c->cells, c->p.bc_y != LBM_BC_BOUNCEBACK, U, R);
    const cudaError_t e = c->tile_buf.upload(list.items, list.nbr);
    if (e == cudaErrorMemoryAllocation) {   // no room: a launch a step
        c->tile = nullptr;
        return LBM_OK;
    }
    if (e != cudaSuccess) return LBM_ECUDA;
    c->tile_items = (int)list.items.size();
    c->tile_grid = c->tile_items;
    while ((1 << c->tile_ulog) < U) ++c->tile_ulog;
    return LBM_OK;
}

// Queues one step.
cudaError_t sp_step_once(lbm_sp_ctx* c) {
    const void* in = c->g[c->cur];
    void* out = c->g[1 - c->cur];
    int N = (int)c->N;
    void* k = c->form == LBM_F64 ? (void*)&c->K : (void*)&c->kf;
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
// counters and the abort flag; wait_extra / wait_limit as in StepArgs.
cudaError_t sp_step_tiles(lbm_sp_ctx* c, int n, int wait_extra = 0, int wait_limit = lbm::kWaitLimit) {
    SpTileArgs a;
    a.g0 = c->g[c->cur];
    a.g1 = c->g[1 - c->cur];
    a.src = c->src;
    a.uprev = c->ufield;
    a.N = (int)c->N;
    a.nitems = c->tile_items;
    a.nsteps = n;
    a.ulog = c->tile_ulog;
    a.wait_limit = wait_limit;
    a.wait_extra = wait_extra;
    a.work = c->tile_buf.work;
    a.nbr = c->tile_buf.nbr;
    a.done = c->tile_buf.done;
    a.status = c->d_status;
    if (n > 1) {
        const cudaError_t e = cudaMemsetAsync(a.done, 0, ((size_t)c->tile_items + 1) * sizeof(int), c->stream);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {&a, c->form == LBM_F64 ? (void*)&c->K : (void*)&c->kf};
    c->cur ^= n & 1;
    // one step: no block waits, so the grid need not be resident at once
    return n > 1 ? cudaLaunchCooperativeKernel(c->tile, dim3(c->tile_grid), dim3(kSpThreads), args, 0, c->stream)
                 : cudaLaunchKernel(c->tile, dim3(c->tile_grid), dim3(kSpThreads), args, 0, c->stream);
}

// After a synchronisation: a bounded wait of the tiles that ran out.
lbm_status sp_device_status(lbm_sp_ctx* c) {
    if (!c->tile) return LBM_OK;
    int st = 0;
    cudaError_t r = cudaMemcpyAsync(&st, c->d_status, sizeof(int), cudaMemcpyDeviceToHost, c->stream);
    if (r == cudaSuccess) r = cudaStreamSynchronize(c->stream);
    if (r != cudaSuccess) return sp_cuda(c, r, "status read-back");
    return st == 0 ? LBM_OK : sp_fail(c, LBM_ETIMEOUT, "a bounded device wait ran out in the step kernel");
}

template <typename R>
void sp_fields(lbm_sp_ctx* c, const SpConst<R>& K, unsigned mask) {
    const R *g = static_cast<const R*>(c->g[c->cur]), *src = static_cast<const R*>(c->src);
    const int n = blocks(c->N);
    switch (c->kind) {
        case 1: sp1_fields_kernel<1, R><<<n, 256, 0, c->stream>>>(g, src, c->N, K, c->p.p0, mask, c->d_tmp); break;
        case 2: sp1_fields_kernel<2, R><<<n, 256, 0, c->stream>>>(g, src, c->N, K, c->p.p0, mask, c->d_tmp); break;
        case 4: sp_fields_kernel<true, R><<<n, 256, 0, c->stream>>>(g, src, c->N, K, mask, c->d_tmp); break;
        default: sp_fields_kernel<false, R><<<n, 256, 0, c->stream>>>(g, src, c->N, K, mask, c->d_tmp);
    }
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
    c->K = SpConst<double>{p.nx, p.ny, p.bc_y == LBM_BC_BOUNCEBACK ? 1 : 0, 1.0 / tau, 1.0 - 0.5 / tau, tau - 0.5,
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
        const int n = c->tile ? std::min(nsteps - s, lbm::kLaunchSteps) : 1;
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
    const bool m1 = c->p.model == LBM_SP_NEARLY_INCOMPRESSIBLE;
    const unsigned ok = LBM_FIELD_UX | LBM_FIELD_UY | LBM_FIELD_P | (m1 ? LBM_FIELD_RHO : 0u);
    if (!host_out || mask == 0 || (mask & ~ok)) return sp_fail(c, LBM_EINVAL, "bad mask or output");
    if (!c->ready) return sp_fail(c, LBM_ESTATE, "not initialised");
    const int nf = ((mask & LBM_FIELD_UX) ? 1 : 0) + ((mask & LBM_FIELD_UY) ? 1 : 0) + ((mask & LBM_FIELD_P) ? 1 : 0) +
                   ((mask & LBM_FIELD_RHO) ? 1 : 0);
    if (c->form == LBM_F64) sp_fields(c, c->K, mask);
    else sp_fields(c, c->kf, mask);
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

lbm_status lbm_sp_inject_wait_timeout(lbm_sp_ctx* c, int rounds) {
    if (!c) return LBM_EINVAL;
    if (rounds < 1 || rounds > lbm::kWaitLimit) return sp_fail(c, LBM_EINVAL, "rounds must be in 1 .. 2^21");
    if (!c->ready) return sp_fail(c, LBM_ESTATE, "not initialised");
    if (!c->tile) return sp_fail(c, LBM_ESTATE, "the context runs a launch a step");
    const cudaError_t e = sp_step_tiles(c, 2, 1, rounds);   // every wait of the second step runs out
    return e == cudaSuccess ? LBM_OK : sp_cuda(c, e, "step kernel");
}

const char* lbm_sp_last_error(const lbm_sp_ctx* c) { return c ? c->err.c_str() : "null context"; }

void lbm_sp_destroy(lbm_sp_ctx* c) {
    if (!c) return;
    sp_release(c);
    delete c;
}

}  // extern "C"
