// Discrete adjoint of the fused step with checkpoint-and-recompute.
//
// Objectives (Sec. 3, Figs. 10-12: time-integrated wall loads) over the states
// n = 0 .. N-1 that N steps read:
//   J_tau = sum_n sum_x (tau_w,bottom + tau_w,top),
//   J_p   = sum_n sum_x (p_w,bottom + p_w,top),
// at interior columns, tau_w = rho_1 nu (9 v_1 - v_2) / 3 and
// p_w = k^2 p0(rho_1) - kappa rho_1 lap(rho) - (kappa/2)|grad rho|^2 (Eq. 2.4).
// The adjoint recursion is lambda^N = 0,
//   lambda^n = (d f^{n+1} / d f^n)^T lambda^{n+1} + (d J_n / d f^n)^T,
// the exact transpose of the linearised step that lbm_step takes: moments,
// ghost densities, EOS potential, Laplacian, force (Eq. 2.17), velocity-shift
// BGK or MRT collision, pressure columns, bounce-back streaming. Where the pressure
// column's phase weight is clamped its derivative is taken as zero (the
// derivative almost everywhere). Gradients:
//   dJ/drho0(x) = sum_i w_i lambda^0_i(x)          (f^0 = f_eq(rho0, 0)),
//   dJ/d(dp)    through the column densities, d rho_root / d p = 1 / (k^2 p0'),
//   dJ/dG       = sum_n sum_x Fbar(x)              (body force in F).
//
// One reverse step is two gather-only kernels (no atomics, so results do not
// depend on scheduling): the local transpose per node, and the transposed
// stencils per tile. The forward states of each block of K steps are recomputed
// from a checkpoint by the forward context, in place of their storage; their
// fields, which the reverse chain reads, are computed for many states per
// launch. The reverse arithmetic is FP64, or FP32 on request (lbm_adjoint_set_precision);
// sums over steps are FP64 either way.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "lbm.h"
#include "lbm_internal.h"
#include "lbm_kernels.cuh"

namespace {

using lbm::ex_;
using lbm::ey_;
using lbm::opp_;

// T: the reverse sweep's arithmetic type (double, or float where the forward
// is FP32 and the gradient's bound is far above FP32 rounding)
template <typename T>
__device__ __forceinline__ T wq(int i) { return lbm::w_<T>(i); }

template <typename T>
struct AdjGeo {
    int nx, ny, walls, bc_x;
    int fp;                       // plane pitch of a stored state: rows of nine planes, f[(y * 9 + i) * fp + x]
    int eos_kind;                 // 0 Carnahan-Starling, 1 Peng-Robinson
    T RT, a, b4, k2, kappa, tau, inv_tau, nu, wet, gx, gy;
    T bpr, aalpha;                // PR: b and a alpha(T)
    T g_in, l_in, g_out, l_out, ph_g, inv_dph;  // inv_dph = 0: single phase, no blend
    T w_tau, w_p;
    // collision: BGK (mrt = 0) or MRT with rates over the squared row norms of
    // the moment basis (mrate[k] = s_k / |M_k|^2); the equilibrium velocity is
    // u + ushift F / rho with ushift = tau (BGK) or 1 / s_j (MRT)
    int mrt;
    T ushift, mrate[9];
};

// the FP64 parameters rounded to the reverse sweep's type
template <typename T>
AdjGeo<T> geo_as(const AdjGeo<double> &d)
{
    AdjGeo<T> g;
    g.nx = d.nx; g.ny = d.ny; g.walls = d.walls; g.bc_x = d.bc_x; g.fp = d.fp; g.eos_kind = d.eos_kind;
    g.RT = (T)d.RT; g.a = (T)d.a; g.b4 = (T)d.b4; g.k2 = (T)d.k2; g.kappa = (T)d.kappa; g.tau = (T)d.tau;
    g.inv_tau = (T)d.inv_tau; g.nu = (T)d.nu; g.wet = (T)d.wet; g.gx = (T)d.gx; g.gy = (T)d.gy;
    g.bpr = (T)d.bpr; g.aalpha = (T)d.aalpha;
    g.g_in = (T)d.g_in; g.l_in = (T)d.l_in; g.g_out = (T)d.g_out; g.l_out = (T)d.l_out;
    g.ph_g = (T)d.ph_g; g.inv_dph = (T)d.inv_dph; g.w_tau = (T)d.w_tau; g.w_p = (T)d.w_p;
    g.mrt = d.mrt; g.ushift = (T)d.ushift;
    for (int k = 0; k < 9; ++k) g.mrate[k] = (T)d.mrate[k];
    return g;
}

// Lallemand-Luo moment basis (rho, e, eps, j_x, q_x, j_y, q_y, p_xx, p_xy)
// over the D2Q9 velocities: entry (k, i) per class of velocity (rest, axis,
// diagonal), folded at compile time inside unrolled loops.
__device__ __forceinline__ constexpr int mrow(int k, int i)
{
    return k == 0 ? 1
         : k == 1 ? (i == 0 ? -4 : (i <= 4 ? -1 : 2))
         : k == 2 ? (i == 0 ? 4 : (i <= 4 ? -2 : 1))
         : k == 3 ? ex_(i)
         : k == 4 ? ex_(i) * (i <= 4 ? -2 : 1)
         : k == 5 ? ey_(i)
         : k == 6 ? ey_(i) * (i <= 4 ? -2 : 1)
         : k == 7 ? ex_(i) * ex_(i) - ey_(i) * ey_(i)
         : ex_(i) * ey_(i);
}

// t += c v for a small integer constant c (no operation for c = 0)
template <typename T>
__device__ __forceinline__ void acc_c(T &t, int c, T v)
{
    if (c == 1) t += v;
    else if (c == -1) t -= v;
    else if (c != 0) t = fma((T)c, v, t);
}

// v -> K v with K = M^-1 S M = M^T diag(s_k / |M_k|^2) M. K is symmetric, so
// the same map transposes the MRT relaxation f* = f - K (f - f_eq).
template <typename T>
__device__ __forceinline__ void mrt_apply(const AdjGeo<T> &g, const T (&v)[9], T (&out)[9])
{
    T m[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        T t = 0;
#pragma unroll
        for (int i = 0; i < 9; ++i) acc_c(t, mrow(k, i), v[i]);
        m[k] = t * g.mrate[k];
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        T t = 0;
#pragma unroll
        for (int k = 0; k < 9; ++k) acc_c(t, mrow(k, i), m[k]);
        out[i] = t;
    }
}

template <typename T>
__device__ __forceinline__ bool solid_row(const AdjGeo<T> &g, int y) { return g.walls && (y == 0 || y == g.ny - 1); }
template <typename T>
__device__ __forceinline__ bool pcol(const AdjGeo<T> &g, int x) { return g.bc_x && (x == 0 || x == g.nx - 1); }
__device__ __forceinline__ int pmod(int a, int n)
{
    int r = a % n;
    return r < 0 ? r + n : r;
}

// EOS p0 and dp0/drho: Carnahan-Starling (eta = b rho / 4) or Peng-Robinson
// (x = b rho, D = 1 + 2x - x^2).
template <typename T>
__device__ __forceinline__ T cs_p0(const AdjGeo<T> &g, T r)
{
    if (g.eos_kind == 1) {
        const T x = g.bpr * r;
        return r * g.RT / (T(1) - x) - g.aalpha * r * r / (T(1) + x * (T(2) - x));
    }
    const T eta = g.b4 * r, om = T(1) - eta;
    return r * g.RT * (T(1) + eta * (T(1) + eta * (T(1) - eta))) / (om * om * om) - g.a * r * r;
}
template <typename T>
__device__ __forceinline__ T cs_dp0(const AdjGeo<T> &g, T r)
{
    if (g.eos_kind == 1) {
        const T x = g.bpr * r, om = T(1) - x, D = T(1) + x * (T(2) - x);
        return g.RT / (om * om) - T(2) * g.aalpha * r * (T(1) + x) / (D * D);
    }
    const T eta = g.b4 * r, om = T(1) - eta, om2 = om * om;
    return g.RT * (T(1) + eta * (T(4) + eta * (T(4) + eta * (T(-4) + eta)))) / (om2 * om2) - T(2) * g.a * r;
}
template <typename T>
__device__ __forceinline__ T phi_of(const AdjGeo<T> &g, T r) { return g.k2 * cs_p0(g, r) - r / T(3); }

template <typename T>
__device__ __forceinline__ int map_y(const AdjGeo<T> &g, int y)
{
    if (g.walls) return y <= 0 ? 1 - y : (y >= g.ny - 1 ? 2 * g.ny - 3 - y : y);
    return pmod(y, g.ny);
}
template <typename T>
__device__ __forceinline__ int map_x(const AdjGeo<T> &g, int x)
{
    if (g.bc_x) return x < 0 ? 0 : (x > g.nx - 1 ? g.nx - 1 : x);
    return pmod(x, g.nx);
}
// Density seen by a stencil at (x, y), up to two nodes outside the lattice:
// mirror images behind walls (plus the wetting offset), clamp beyond pressure
// columns, wrap on periodic axes.
template <typename T>
__device__ __forceinline__ T ghost_rho(const AdjGeo<T> &g, const T *rho, int x, int y)
{
    const bool beyond = g.walls && (y <= 0 || y >= g.ny - 1);
    return rho[map_y(g, y) * g.nx + map_x(g, x)] + (beyond ? g.wet : T(0));
}

// Phase weight of a pressure column whose neighbour has density rf, and its
// derivative (zero where clamped).
template <typename T>
__device__ __forceinline__ T col_theta(const AdjGeo<T> &g, T rf, T &dth)
{
    dth = 0;
    if (!(g.inv_dph > T(0))) return 0;
    T th = (rf - g.ph_g) * g.inv_dph;
    if (th < T(0)) return 0;
    if (th > T(1)) return 1;
    if (th > T(0) && th < T(1)) dth = g.inv_dph;
    return th;
}

// gx, gy += 3 w_i e_i v: direction i's term of the lattice gradient, zero
// components skipped (i is a constant inside unrolled loops)
template <typename T>
__device__ __forceinline__ void grad_term(T &gx, T &gy, int i, T v)
{
    if (ex_(i) != 0) gx += T(3) * wq<T>(i) * T(ex_(i)) * v;
    if (ey_(i) != 0) gy += T(3) * wq<T>(i) * T(ey_(i)) * v;
}

// ---- stencil pieces ---------------------------------------------------------

// FP64 is bound by the number of FP64 instructions: its stencils add before
// they scale. FP32 is not bound by arithmetic, and its sums over many nodes and
// steps (J, dJ/d dp) show any change of rounding: its stencils add weighted
// terms one by one in direction order. (adj_finish, which FP32 takes without
// pressure columns or without walls, is written in the FP64 form for both; its FP32
// gradients are as far from the FP64 sweep's as with the terms one by one.)
template <typename T>
constexpr bool BY_TERMS = sizeof(T) == 4;

// 3 x 3 neighbourhood of point (c, r) of a shared array with row pitch SW.
template <typename T>
struct Nb {
    T mw, mc, me, zw, zc, ze, pw, pc, pe;  // rows below (m), at (z), above (p)
};
template <int SW, typename T>
__device__ __forceinline__ Nb<T> nb_of(const T *a, int c, int r)
{
    const T *z = a + r * SW + c, *m = z - SW, *p = z + SW;
    return Nb<T>{m[-1], m[0], m[1], z[-1], z[0], z[1], p[-1], p[0], p[1]};
}
// 12 x the lattice gradient 3 sum_i w_i e_i psi(x + e_i) (weights 1/3 and 1/12)
template <typename T>
__device__ __forceinline__ T dx12(const Nb<T> &n) { return T(4) * (n.ze - n.zw) + ((n.me - n.mw) + (n.pe - n.pw)); }
template <typename T>
__device__ __forceinline__ T dy12(const Nb<T> &n) { return T(4) * (n.pc - n.mc) + ((n.pw - n.mw) + (n.pe - n.me)); }
// 6 x lap psi = 36 sum_i w_i (psi(x + e_i) - psi(x))
template <typename T>
__device__ __forceinline__ T lap6(const Nb<T> &n)
{
    const T e = (n.zw + n.ze) + (n.mc + n.pc), k = (n.mw + n.me) + (n.pw + n.pe);
    return T(4) * e + (k - T(20) * n.zc);
}
// grad psi and lap psi at the point a[0] of a shared array with row pitch SW
template <int SW, typename T>
__device__ __forceinline__ void grad_at(const T *a, T &gx, T &gy)
{
    if constexpr (BY_TERMS<T>) {
        gx = gy = 0;
#pragma unroll
        for (int i = 1; i < 9; ++i) grad_term(gx, gy, i, a[ey_(i) * SW + ex_(i)]);
    } else {
        const Nb<T> n = nb_of<SW>(a, 0, 0);
        gx = dx12(n) * T(1.0 / 12.0);
        gy = dy12(n) * T(1.0 / 12.0);
    }
}
template <int SW, typename T>
__device__ __forceinline__ T lap_at(const T *a)
{
    if constexpr (BY_TERMS<T>) {
        T s = 0;
#pragma unroll
        for (int i = 1; i < 9; ++i) s += T(6) * wq<T>(i) * (a[ey_(i) * SW + ex_(i)] - a[0]);
        return s;
    } else {
        return lap6(nb_of<SW>(a, 0, 0)) * T(1.0 / 6.0);
    }
}

// grad rho at a node, ghost densities included
template <typename T>
__device__ __forceinline__ void grad_rho(const AdjGeo<T> &g, const T *rho, int x, int y, T &gx, T &gy)
{
    gx = gy = 0;
#pragma unroll
    for (int i = 1; i < 9; ++i) grad_term(gx, gy, i, ghost_rho(g, rho, x + ex_(i), y + ey_(i)));
}

// ---- forward recompute of the fields of stored states -------------------------

// Values kept per node of a state for the reverse sweep (planes of nx ny):
// density, 1 / density, the equilibrium velocity u_eq = (j + ushift F) / rho (j
// until the force is known), grad L, phi and dphi/drho = k^2 p0' - 1/3;
// and, at the rows next to a wall and the columns next to a pressure column
// only, v = (j + F / 2) (1 / rho) and L, and next to a wall v_x as a quotient (the
// objective's form).
enum { F_RHO, F_IR, F_UX, F_UY, F_LX, F_LY, F_PHI, F_DPHI, F_VX, F_VY, F_LAP, F_VQ, NFIELD };

// Stored state m of a block: state 0 is the checkpoint, the others follow one
// another `stride` bytes apart.
struct States {
    const char *ck, *blk;
    size_t stride;
    template <typename S>
    __device__ __forceinline__ const S *at(int m) const
    {
        return reinterpret_cast<const S *>(m == 0 ? ck : blk + (size_t)m * stride);
    }
};

// A stored value in the sweep's type. FP32 to FP64 by integer operations: the
// conversion instruction runs on the FP64 pipe (1/64 of the FP32 rate), which
// bounds the sweep, and nine of them per node were a tenth of the fields' work.
template <typename T, typename S>
__device__ __forceinline__ T widen(S v) { return (T)v; }
template <>
__device__ __forceinline__ double widen<double>(float v)
{
    const unsigned b = __float_as_uint(v), e = b & 0x7f800000u;
    if (e - 0x00800000u <= 0x7f000000u - 0x00800000u)  // a normal number: rebias the exponent
        return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
    return (double)v;
}

// density of a node of a stored state (populations added in index order)
template <typename S, typename T>
__device__ __forceinline__ T sum9(const S *fr, int fp)
{
    T r = widen<T>(fr[0]);
#pragma unroll
    for (int i = 1; i < 9; ++i) r += widen<T>(fr[i * fp]);
    return r;
}

// Density seen by a stencil of state f at (x, y), up to two nodes outside the
// lattice: mirror images behind walls (plus the wetting offset), the column
// density at and beyond pressure columns, wrap on periodic axes.
template <typename S, typename T>
__device__ __forceinline__ T ext_density(const AdjGeo<T> &g, const S *f, int x, int y)
{
    const bool beyond = g.walls && (y <= 0 || y >= g.ny - 1);
    const S *fr = f + (size_t)map_y(g, y) * 9 * g.fp;
    const int xx = map_x(g, x);
    T r;
    if (pcol(g, xx)) {
        r = sum9<S, T>(fr + (xx == 0 ? 1 : g.nx - 2), g.fp);
        T dth;
        const T th = col_theta(g, r, dth), gg = xx == 0 ? g.g_in : g.g_out, ll = xx == 0 ? g.l_in : g.l_out;
        r = gg + th * (ll - gg);
    } else {
        r = sum9<S, T>(fr + xx, g.fp);
    }
    return beyond ? r + g.wet : r;
}

// 1 / r, phi(r) and dphi/dr. FP64 takes one division for both reciprocals of
// the Carnahan-Starling form (a division is about ten FP64 instructions).
template <typename T>
__device__ __forceinline__ void eos_all(const AdjGeo<T> &g, T r, T &ir, T &phi, T &dphi)
{
    if (BY_TERMS<T> || g.eos_kind == 1) {
        ir = T(1) / r;
        phi = phi_of(g, r);
        dphi = g.k2 * cs_dp0(g, r) - T(1) / T(3);
        return;
    }
    const T eta = g.b4 * r, om = T(1) - eta, om2 = om * om, om3 = om2 * om;
    const T i = T(1) / (r * om3), i3 = i * r;
    ir = i * om3;
    const T p0 = r * g.RT * (T(1) + eta * (T(1) + eta * om)) * i3 - g.a * r * r;
    const T dp0 = g.RT * (T(1) + eta * (T(4) + eta * (T(4) + eta * (T(-4) + eta)))) * (i3 * i3 * om2) - T(2) * g.a * r;
    phi = g.k2 * p0 - r * T(1.0 / 3.0);
    dphi = g.k2 * dp0 - T(1.0 / 3.0);
}

// Tiles of the stencil kernels: TX columns by th rows, one node per thread.
// The host picks th (at most TMAX) so that the tiles fill whole waves of the
// SMs: the FP64 kernels are bound by each SM's FP64 pipe, and 256 tiles of 8
// rows on 152 SMs left a third of it idle.
constexpr int TX = 32, TMAX = 16;
constexpr int AW = TX + 4, BW = TX + 2;  // with two nodes, one node around
constexpr int SMEM_A = AW * (TMAX + 4), SMEM_B = BW * (TMAX + 2);

// Local coordinates of halo point h of a ring of width D around a tile
// (columns -D .. TX+D-1, rows -D .. th+D-1): the rows above and below, then the sides.
template <int D>
__device__ __forceinline__ void halo_point(int th, int h, int &c, int &r)
{
    constexpr int W = TX + 2 * D;
    if (h < 2 * D * W) {
        const int q = h / W;
        c = h - q * W - D;
        r = q < D ? q - D : th + q - D;
    } else {
        h -= 2 * D * W;
        const int q = h / (2 * D), k = h - q * 2 * D;
        r = q;
        c = k < D ? k - D : TX + k - D;
    }
}
template <int D>
__device__ __forceinline__ int halo_count(int th) { return (TX + 2 * D) * (th + 2 * D) - TX * th; }

// The fields of states m0 + blockIdx.y of a block, one launch for many states:
// they do not depend on the adjoint, so they come off the reverse sweep's
// serial chain and fill the GPU together. Two passes: per node (density,
// momentum, equation of state), then the stencils per tile, so that no ghost
// point repeats the sums and the equation of state of its node.
template <typename S, typename T>
__global__ void __launch_bounds__(128) adj_nodes(AdjGeo<T> g, States st, int m0, T *out)
{
    const int c = blockIdx.x * 128 + threadIdx.x;
    if (c >= g.nx * g.ny) return;
    const int y = c / g.nx, x = c - y * g.nx;
    if (solid_row(g, y)) return;
    const size_t n = (size_t)g.nx * g.ny;
    T *o = out + (size_t)blockIdx.y * NFIELD * n + c;
    const bool col = pcol(g, x);
    const S *fr = st.at<S>(m0 + blockIdx.y) + (size_t)y * 9 * g.fp + (col ? (x == 0 ? 1 : g.nx - 2) : x);
    T v[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = widen<T>(fr[i * g.fp]);
    T r = v[0];
#pragma unroll
    for (int i = 1; i < 9; ++i) r += v[i];
    if (col) {
        T dth;
        const T th = col_theta(g, r, dth), gg = x == 0 ? g.g_in : g.g_out, ll = x == 0 ? g.l_in : g.l_out;
        r = gg + th * (ll - gg);
    }
    T ir, phi, dphi;
    eos_all(g, r, ir, phi, dphi);
    o[F_RHO * n] = r;
    o[F_PHI * n] = phi;
    o[F_DPHI * n] = dphi;
    if (col) return;
    o[F_IR * n] = ir;
    T X = 0, Y = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        acc_c(X, ex_(i), v[i]);
        acc_c(Y, ey_(i), v[i]);
    }
    o[F_UX * n] = X;
    o[F_UY * n] = Y;
}

template <typename T>
__global__ void __launch_bounds__(TX * TMAX) adj_forces(AdjGeo<T> g, int th, T *out)
{
    __shared__ T R[SMEM_A], P[SMEM_B], L[SMEM_B];
    const int tid = threadIdx.x, tx = tid & (TX - 1), ty = tid / TX, tn = TX * th;
    const int ntx = (g.nx + TX - 1) / TX, by = blockIdx.x / ntx;
    const int x0 = (blockIdx.x - by * ntx) * TX, y0 = (g.walls ? 1 : 0) + by * th;
    const int x = x0 + tx, y = y0 + ty;
    const size_t n = (size_t)g.nx * g.ny;
    T *o = out + (size_t)blockIdx.y * NFIELD * n;
    const int ymax = g.walls ? g.ny - 2 : g.ny - 1;  // last fluid row
    const bool node = x < g.nx && y <= ymax && !pcol(g, x);

    // densities of the tile and two nodes around it, phi one node around
    auto load = [&](int c, int r) {
        const int gx = x0 + c, gy = y0 + r;
        T v = T(1), ph = T(0);
        if (gx < g.nx + 2 && gy <= ymax + 2) {
            const size_t q = (size_t)map_y(g, gy) * g.nx + map_x(g, gx);
            v = o[F_RHO * n + q];
            const bool beyond = g.walls && (gy <= 0 || gy >= g.ny - 1) && g.wet != T(0);
            if (beyond) v += g.wet;
            if (c >= -1 && c <= TX && r >= -1 && r <= th) ph = beyond ? phi_of(g, v) : o[F_PHI * n + q];
        }
        R[(r + 2) * AW + c + 2] = v;
        if (c >= -1 && c <= TX && r >= -1 && r <= th) P[(r + 1) * BW + c + 1] = ph;
    };
    load(tx, ty);
    for (int h = tid; h < halo_count<2>(th); h += tn) {
        int c, r;
        halo_point<2>(th, h, c, r);
        load(c, r);
    }
    T X = 0, Y = 0, ir = 0;
    const size_t c = (size_t)y * g.nx + x;
    if (node) {
        X = o[F_UX * n + c];
        Y = o[F_UY * n + c];
        ir = o[F_IR * n + c];
    }
    __syncthreads();
    const T lap = lap_at<AW>(R + (ty + 2) * AW + tx + 2);
    L[(ty + 1) * BW + tx + 1] = lap;
    for (int h = tid; h < halo_count<1>(th); h += tn) {
        int k, q;
        halo_point<1>(th, h, k, q);
        L[(q + 1) * BW + k + 1] = lap_at<AW>(R + (q + 2) * AW + k + 2);
    }
    __syncthreads();
    if (!node) return;
    const T r = R[(ty + 2) * AW + tx + 2];
    const int k = (ty + 1) * BW + tx + 1;
    T gpx, gpy, glx, gly;
    grad_at<BW>(P + k, gpx, gpy);
    grad_at<BW>(L + k, glx, gly);
    const T FX = -gpx + g.kappa * r * glx + g.gx, FY = -gpy + g.kappa * r * gly + g.gy;
    o[F_UX * n + c] = (X + g.ushift * FX) * ir;
    o[F_UY * n + c] = (Y + g.ushift * FY) * ir;
    o[F_LX * n + c] = glx;
    o[F_LY * n + c] = gly;
    const bool edge = g.bc_x && (x == 1 || x == g.nx - 2);
    if (edge || (g.walls && (y <= 2 || y >= g.ny - 3))) {
        o[F_VX * n + c] = (X + T(0.5) * FX) * ir;
        o[F_VY * n + c] = (Y + T(0.5) * FY) * ir;
        o[F_LAP * n + c] = lap;
        o[F_VQ * n + c] = (X + T(0.5) * FX) / r;
    }
}

// Wall shear and wall pressure of states m0 + blockIdx.z at the columns of one
// wall (blockIdx.y): out[z][0 .. 2 nx) = tau_w, [2 nx .. 4 nx) = p_w (bottom
// then top), zero at pressure columns. Only the wall's own rows are read: the
// densities of rows -1 .. 4 counted from the wall (six rows, ghosts among
// them) give the Laplacian and phi of four and the force of two. J sums terms
// of both signs over all columns and steps, so in FP32 the constants' rounding
// shows in it: the weights are applied term by term.
constexpr int LT = 64;  // columns of a block
template <typename S, typename T>
__global__ void __launch_bounds__(128) adj_loads(AdjGeo<T> g, States st, int m0, double *out)
{
    constexpr int EW = LT + 4, PW = LT + 2;
    __shared__ T E[6 * EW], P[4 * PW], L[4 * PW], J[2 * LT], F[2 * LT];
    const int x0 = blockIdx.x * LT, side = blockIdx.y, tid = threadIdx.x;
    const int up = side ? -1 : 1;  // row j of E is lattice row j - 1, or ny - j
    const S *f = st.at<S>(m0 + blockIdx.z);
    for (int k = tid; k < 6 * EW; k += 128) {
        const int j = k / EW, x = x0 + k % EW - 2, y = side ? g.ny - j : j - 1;
        E[k] = x < g.nx + 2 ? ext_density<S, T>(g, f, x, y) : T(1);
    }
    {
        const int j = tid / LT, x = x0 + tid % LT, y = side ? g.ny - 2 - j : 1 + j;
        T X = 0;
        if (x < g.nx) {
            const S *fr = f + (size_t)y * 9 * g.fp + x;
#pragma unroll
            for (int i = 0; i < 9; ++i) acc_c(X, ex_(i), widen<T>(fr[i * g.fp]));
        }
        J[tid] = X;
    }
    __syncthreads();
    for (int k = tid; k < 4 * PW; k += 128) {
        const int j = k / PW, c = k % PW;
        const T *e = E + (j + 1) * EW + c + 1;
        const T e0 = e[0];
        T s = 0;
#pragma unroll
        for (int i = 1; i < 9; ++i) s += T(6) * wq<T>(i) * (e[up * ey_(i) * EW + ex_(i)] - e0);
        P[k] = phi_of(g, e0);
        L[k] = s;
    }
    __syncthreads();
    // F_x of rows 1 and 2
    {
        const int j = tid / LT, c = tid % LT;
        T gpx = 0, glx = 0, unused = 0;
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            if (ex_(i) == 0) continue;
            const int q = (j + 1 + up * ey_(i)) * PW + c + 1 + ex_(i);
            grad_term(gpx, unused, i, P[q]);
            grad_term(glx, unused, i, L[q]);
        }
        F[tid] = -gpx + g.kappa * E[(j + 2) * EW + c + 2] * glx + g.gx;
    }
    __syncthreads();
    const int c = tid & (LT - 1), x = x0 + c;
    if (x >= g.nx) return;
    double *o = out + (size_t)blockIdx.z * 4 * g.nx + side * g.nx + x;
    const bool col = pcol(g, x);
    const T *e = E + 2 * EW + c + 2;
    const T r1 = e[0];
    if (tid < LT) {
        const T m1 = J[c] + T(0.5) * F[c], v2 = (J[LT + c] + T(0.5) * F[LT + c]) / e[EW];
        o[0] = col ? 0.0 : (double)(g.nu * (T(9) * m1 - r1 * v2) / T(3));
    } else {
        T grx = 0, gry = 0;
#pragma unroll
        for (int i = 1; i < 9; ++i) grad_term(grx, gry, i, e[up * ey_(i) * EW + ex_(i)]);
        o[2 * g.nx] = col ? 0.0
                          : (double)(g.k2 * cs_p0(g, r1) - g.kappa * r1 * L[PW + c + 1] -
                                     T(0.5) * g.kappa * (grx * grx + gry * gry));
    }
}

// acc[t] += out[0][t] + out[1][t] + ..., in state order
__global__ void adj_add_loads(const double *__restrict__ out, int len, int m, double *acc)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= len) return;
    double a = acc[t];
    for (int k = 0; k < m; ++k) a += out[(size_t)k * len + t];
    acc[t] = a;
}

// ---- reverse step -----------------------------------------------------------

// The moments sum a_i, sum e_i a_i, sum e_i e_i a_i of a_i = w_i scale v_i.
template <typename T>
struct Mom {
    T m0, mx, my, mxx, myy, mxy;
};
template <typename T>
__device__ __forceinline__ Mom<T> weighted_moments(const T (&v)[9], T scale)
{
    Mom<T> m;
    if constexpr (BY_TERMS<T>) {
        m = Mom<T>{0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const T a = wq<T>(i) * (v[i] * scale);
            m.m0 += a;
            acc_c(m.mx, ex_(i), a);
            acc_c(m.my, ey_(i), a);
            acc_c(m.mxx, ex_(i) * ex_(i), a);
            acc_c(m.myy, ey_(i) * ey_(i), a);
            acc_c(m.mxy, ex_(i) * ey_(i), a);
        }
    } else {
        // the weights applied to sums of pairs
        const T w0 = wq<T>(0) * scale, w1 = wq<T>(1) * scale, w5 = wq<T>(5) * scale;
        const T p = w5 * (v[5] + v[7]), q = w5 * (v[6] + v[8]);
        const T a = w5 * (v[5] - v[7]), b = w5 * (v[6] - v[8]);
        const T d = p + q;
        m.mxx = w1 * (v[1] + v[3]) + d;
        m.myy = w1 * (v[2] + v[4]) + d;
        m.mxy = p - q;
        m.mx = w1 * (v[1] - v[3]) + (a - b);
        m.my = w1 * (v[2] - v[4]) + (a + b);
        m.m0 = w0 * v[0] + ((m.mxx + m.myy) - d);
    }
    return m;
}

// Programmatic dependent launch (lbm_rows2.cuh): wait for the kernel before,
// then let the next one's launch overlap this one. A grid may thus be resident
// while the one before still writes its inputs. Those inputs are plain pointers:
// const __restrict__ would promise that they do not change while the grid lives,
// and allow loads from the read-only cache, or ahead of the wait. The state's
// fields (fld) are complete before a run's first grid starts (adj_chain_t).
__device__ __forceinline__ void chain_start()
{
    lbm::griddep_wait();
    lbm::griddep_launch_dependents();
}

// Local part of the reverse step at every fluid node: reverse streaming,
// reverse collision, the pressure column fed by this node, and the wall
// objective terms of this node. Outputs Fbar (A), jbar, the local rho-bar (R;
// a column's own entry is written by its interior neighbour), the wall
// pressure's gradient sources of the rows next to the walls (Cw[side][x, y][nx])
// and, with PART (MRT, or tau != 1, where it is not zero), f*-bar - K f*-bar
// into lam_out; Fbar is also added to its FP64 per-node sum over the steps (AS).
//
// FP64 is bound by the FP64 pipe, so the state's fields are read instead of
// recomputed and the weights apply to sums of populations. The `eblocks` first
// blocks take the nodes next to the pressure columns (2 ny of them), whose
// work is three times a node's: spread one lane per warp over the lattice they
// would slow two of every sixteen warps of a 512-wide row, always on the same
// SMs (51k cycles on the busiest SM against 29k on average).
template <typename T, bool PART, int BLOCK>
__global__ void __launch_bounds__(BLOCK) adj_local(AdjGeo<T> g, int eblocks, const T *lam_in,
                                                   const T *__restrict__ fld, T *lam_out, T *Ax, T *Ay,
                                                   T *Jbx, T *Jby, T *R, T *Cw, double *AS)
{
    chain_start();
    const int n = g.nx * g.ny;
    const bool edge = (int)blockIdx.x < eblocks;  // uniform
    int x, y;
    if (edge) {
        const int k = blockIdx.x * BLOCK + threadIdx.x;
        if (k >= 2 * g.ny) return;
        y = k >= g.ny ? k - g.ny : k;
        x = k >= g.ny ? g.nx - 2 : 1;
    } else {
        const int k = (blockIdx.x - eblocks) * BLOCK + threadIdx.x;
        if (k >= n) return;
        y = k / g.nx;
        x = k - y * g.nx;
        if (g.bc_x && (x == 1 || x == g.nx - 2)) return;
    }
    if (solid_row(g, y) || pcol(g, x)) return;  // their entries stay zero
    const int c = y * g.nx + x;
    const size_t N = n;

    // reverse streaming: f*_i(x) went to x + e_i, or back to x as opp(i)
    int xm = x - 1, xp = x + 1, ym = y - 1, yp = y + 1;
    if (!g.bc_x) { xm = xm < 0 ? g.nx - 1 : xm; xp = xp == g.nx ? 0 : xp; }
    bool bb = false, bt = false;
    if (g.walls) { bb = ym == 0; bt = yp == g.ny - 1; }
    else { ym = ym < 0 ? g.ny - 1 : ym; yp = yp == g.ny ? 0 : yp; }
    const int rz = y * g.nx, rm = ym * g.nx, rp = yp * g.nx;
    T gb[9];
    gb[0] = lam_in[c];
    gb[1] = lam_in[n + rz + xp];
    gb[3] = lam_in[3 * N + rz + xm];
    gb[2] = lam_in[bt ? 4 * N + c : 2 * N + rp + x];
    gb[5] = lam_in[bt ? 7 * N + c : 5 * N + rp + xp];
    gb[6] = lam_in[bt ? 8 * N + c : 6 * N + rp + xm];
    gb[4] = lam_in[bb ? 2 * N + c : 4 * N + rm + x];
    gb[7] = lam_in[bb ? 5 * N + c : 7 * N + rm + xm];
    gb[8] = lam_in[bb ? 6 * N + c : 8 * N + rm + xp];

    const T ux = fld[F_UX * N + c], uy = fld[F_UY * N + c], inv_r = fld[F_IR * N + c];
    const T glx = fld[F_LX * N + c], gly = fld[F_LY * N + c];

    // collision f* = f - K (f - f_eq(rho, u_eq)), K = I / tau (BGK) or M^-1 S M
    // (MRT): f-bar = g - K g, f_eq-bar = K g
    T lam[9];
    Mom<T> m;
    if (PART && g.mrt) {
        T kg[9];
        mrt_apply(g, gb, kg);
#pragma unroll
        for (int i = 0; i < 9; ++i) lam[i] = gb[i] - kg[i];
        m = weighted_moments(kg, T(1));
    } else {
        if (PART) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                if constexpr (BY_TERMS<T>) lam[i] = __fsub_rn(gb[i], __fmul_rn(gb[i], g.inv_tau));
                else lam[i] = gb[i] - gb[i] * g.inv_tau;
            }
        }
        m = weighted_moments(gb, g.inv_tau);
    }
    // f_eq_i = w_i rho (1 + 3 e_i.u + 4.5 (e_i.u)^2 - 1.5 u^2) is quadratic in
    // e_i: with s = M u (second moments), u_eq-bar / rho = 3 m + 9 s - 3 u m0
    // and rho-bar - u_eq-bar . u_eq / rho = m0 (1 + 1.5 u^2) - 4.5 u.s
    T rb, jbx, jby;
    if constexpr (BY_TERMS<T>) {
        // every product that is fused is named: the compiler's choice depends on
        // the code around it
        auto dot = [](T a, T b, T c, T d) { return __fmaf_rn(a, b, __fmul_rn(c, d)); };
        const T ux2 = __fmul_rn(ux, ux), uy2 = __fmul_rn(uy, uy), uxy = __fmul_rn(T(2) * ux, uy);
        const T usq = __fadd_rn(ux2, uy2);
        rb = dot(T(3), dot(ux, m.mx, uy, m.my), m.m0, __fmaf_rn(T(-1.5), usq, T(1)));
        rb = __fmaf_rn(T(4.5), __fmaf_rn(uy2, m.myy, dot(ux2, m.mxx, uxy, m.mxy)), rb);
        jbx = __fmaf_rn(-__fmul_rn(T(3), ux), m.m0, dot(T(3), m.mx, T(9), dot(ux, m.mxx, uy, m.mxy)));
        jby = __fmaf_rn(-__fmul_rn(T(3), uy), m.m0, dot(T(3), m.my, T(9), dot(ux, m.mxy, uy, m.myy)));
        rb = __fsub_rn(rb, dot(jbx, ux, jby, uy));
    } else {
        const T sx = ux * m.mxx + uy * m.mxy, sy = ux * m.mxy + uy * m.myy;
        const T usq = ux * ux + uy * uy;
        rb = m.m0 * (T(1) + T(1.5) * usq) - T(4.5) * (ux * sx + uy * sy);
        jbx = T(3) * (m.mx - ux * m.m0) + T(9) * sx;
        jby = T(3) * (m.my - uy * m.m0) + T(9) * sy;
    }
    T ax = g.ushift * jbx, ay = g.ushift * jby;

    // wall objective terms (interior columns; a row may serve both walls on
    // very low channels)
    if (g.walls && (y <= 2 || y >= g.ny - 3)) {
        const T *rho = fld + F_RHO * N;
        for (int side = 0; side < 2; ++side) {
            const int y1 = side ? g.ny - 2 : 1, y2 = side ? g.ny - 3 : 2;
            if (y == y1) {
                const T v2 = fld[F_VQ * N + y2 * g.nx + x];
                jbx += g.w_tau * T(3) * g.nu;
                ax += g.w_tau * T(1.5) * g.nu;
                rb += -g.w_tau * g.nu / T(3) * v2;
                rb += g.w_p * (g.k2 * cs_dp0(g, rho[c]) - g.kappa * fld[F_LAP * N + c]);
                T grx, gry;
                grad_rho(g, rho, x, y, grx, gry);
                Cw[(2 * side) * g.nx + x] = -g.w_p * g.kappa * grx;
                Cw[(2 * side + 1) * g.nx + x] = -g.w_p * g.kappa * gry;
            }
            if (y == y2) {
                const T r1v = rho[y1 * g.nx + x];
                const T v2 = fld[F_VX * N + c];
                jbx += -g.w_tau * g.nu / T(3) * r1v * inv_r;
                ax += -g.w_tau * g.nu / T(6) * r1v * inv_r;
                rb += g.w_tau * g.nu / T(3) * r1v * v2 * inv_r;
            }
        }
    }

    // pressure column fed by this node:
    // f*_i(x_b) = f_eq_i(rho_b, v_f) + (1 - 1/tau)(f_i(x_f) - f_eq_i(rho_f, v_f)),
    // v_f = (j_f + F_f / 2) / rho_f
    if (edge) {
        const T omt = PART ? T(1) - g.inv_tau : T(0);
        const int xb = x == 1 ? 0 : g.nx - 1, cb = y * g.nx + xb;
        T gc[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            int tx = xb + ex_(i), ty = y + ey_(i);
            gc[i] = 0;
            if (g.walls && (ty == 0 || ty == g.ny - 1)) continue;  // into the column's own (unread) slots
            if (!g.walls) ty = pmod(ty, g.ny);
            if (tx < 0 || tx >= g.nx) continue;                      // leaves the lattice
            gc[i] = lam_in[i * N + ty * g.nx + tx];
        }
        const T r = fld[F_RHO * N + c], rbv = fld[F_RHO * N + cb];
        const T vx = fld[F_VX * N + c], vy = fld[F_VY * N + c];
        const T vsq = vx * vx + vy * vy;
        T rbb = 0, vbx = 0, vby = 0;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const T ev = T(ex_(i)) * vx + T(ey_(i)) * vy;
            const T q = wq<T>(i) * (T(1) + T(3) * ev + T(4.5) * ev * ev - T(1.5) * vsq);
            if (PART) lam[i] += omt * gc[i];
            rbb += gc[i] * q;
            if (PART) rb -= omt * gc[i] * q;
            const T s = gc[i] * (rbv - omt * r) * wq<T>(i);
            vbx += s * (T(3 * ex_(i)) + T(9) * ev * T(ex_(i)) - T(3) * vx);
            vby += s * (T(3 * ey_(i)) + T(9) * ev * T(ey_(i)) - T(3) * vy);
        }
        R[cb] = rbb;
        jbx += vbx * inv_r;
        jby += vby * inv_r;
        ax += T(0.5) * vbx * inv_r;
        ay += T(0.5) * vby * inv_r;
        rb -= (vbx * vx + vby * vy) * inv_r;
    }

    // F = ... + kappa rho grad L: the rho factor
    rb += g.kappa * (ax * glx + ay * gly);

    if (PART) {
#pragma unroll
        for (int i = 0; i < 9; ++i) lam_out[i * N + c] = lam[i];
    }
    Ax[c] = ax;
    Ay[c] = ay;
    AS[c] += (double)ax;  // sums over the steps: the body-force sensitivities
    AS[N + c] += (double)ay;
    Jbx[c] = jbx;
    Jby[c] = jby;
    R[c] = rb;
}

// Non-local part of the reverse step, one tile per block: Lbar and phibar
// (transposed gradients of the force), the adjoint of the ghost-extended
// density and its fold onto the lattice, and
// lambda^n_i(x) = (f*-bar - K f*-bar)_i + rhobar + jbar . e_i.
//
// The lattice gradient is odd, so its transpose is minus the divergence:
// Lbar = -div(kappa rho A) + its objective source, phibar = div A, and with the
// symmetric Laplacian Ebar = dphi phibar + lap Lbar - div C. The ghosts fold
// before the next operator instead of after the last one: behind a wall the
// density is mirrored at the half-way plane, so the fold of -div(B) over the
// ghost row is the same divergence with B extended symmetrically in x and
// antisymmetrically in y, and the fold of lap Lbar is the Laplacian with Lbar
// mirrored; a periodic axis wraps; at and beyond a pressure column, whose
// density is one value, Ebar sums into the column's rho-bar, which reaches the
// interior neighbour through the phase weight (its sensitivities are added to
// FP64 sums over the steps, colp). wet != 0 shifts the density at which a
// wall ghost's dphi is taken: phibar of the ghost row is then weighted by
// itself. Five shared arrays and two barriers replace three kernels and five
// arrays in memory: 31 -> 15 us at 512 x 128 in FP64 (the FP64 pipe needs 6;
// the rest is one wave's load, two barriers and the launch).
template <typename T, bool PART>
__global__ void __launch_bounds__(TX * TMAX) adj_finish(AdjGeo<T> g, int th, const T *__restrict__ fld,
                                                        const T *Ax, const T *Ay, const T *Jbx, const T *Jby,
                                                        const T *R, const T *Cw, T *lam_out, double *colp)
{
    __shared__ T SX[SMEM_A], SY[SMEM_A], BX[SMEM_A], BY[SMEM_A], SL[SMEM_B];
    chain_start();
    const int tid = threadIdx.x, tx = tid & (TX - 1), ty = tid / TX, tn = TX * th;
    const int ntx = (g.nx + TX - 1) / TX, by = blockIdx.x / ntx;
    const int x0 = (blockIdx.x - by * ntx) * TX, y0 = (g.walls ? 1 : 0) + by * th;
    const int x = x0 + tx, y = y0 + ty, nx = g.nx, ny = g.ny;
    const size_t N = (size_t)nx * ny;
    const int ymax = g.walls ? ny - 2 : ny - 1;  // last fluid row
    const T *rho = fld + F_RHO * N;

    // Fbar and rho Fbar on the tile and two nodes around it
    auto load = [&](int c, int r) {
        int gx = x0 + c, gy = y0 + r;
        T ax = 0, ay = 0, rv = 0;
        bool in = gx < nx + 2 && gy <= ymax + 2, flip = false;
        if (g.bc_x) in = in && gx >= 1 && gx <= nx - 2;
        else if (in) gx = pmod(gx, nx);
        if (g.walls) {
            in = in && gy >= 0 && gy <= ny - 1;
            flip = gy == 0 || gy == ny - 1;
            gy = gy == 0 ? 1 : (gy == ny - 1 ? ny - 2 : gy);
        } else if (in) {
            gy = pmod(gy, ny);
        }
        if (in) {
            const size_t q = (size_t)gy * nx + gx;
            ax = Ax[q];
            ay = flip ? -Ay[q] : Ay[q];
            rv = rho[q];
        }
        const int k = (r + 2) * AW + c + 2;
        SX[k] = ax;
        SY[k] = ay;
        BX[k] = rv * ax;
        BY[k] = rv * ay;
    };
    load(tx, ty);
    for (int h = tid; h < halo_count<2>(th); h += tn) {
        int c, r;
        halo_point<2>(th, h, c, r);
        load(c, r);
    }
    const bool node = x < nx && y <= ymax && !pcol(g, x);
    const size_t cn = (size_t)y * nx + x;
    T rb = 0, jx = 0, jy = 0, dphi = 0;
    if (node) {
        rb = R[cn];
        jx = Jbx[cn];
        jy = Jby[cn];
        dphi = fld[F_DPHI * N + cn];
    }
    __syncthreads();

    // Lbar on the tile and one node around it (a ghost row repeats its wall row)
    const T kap = g.kappa * T(1.0 / 12.0);
    auto lbar = [&](int c, int r) {
        const int gy = y0 + r;
        int q = r;
        if (g.walls) q = gy < 1 ? 1 - y0 : (gy > ny - 2 ? ny - 2 - y0 : r);
        T s = -kap * (dx12(nb_of<AW>(BX, c + 2, q + 2)) + dy12(nb_of<AW>(BY, c + 2, q + 2)));
        if (g.walls && g.w_p != T(0) && (y0 + q == 1 || y0 + q == ny - 2)) {
            const int gx = g.bc_x ? x0 + c : pmod(x0 + c, nx);
            if (!g.bc_x || (gx >= 1 && gx <= nx - 2)) s -= g.w_p * g.kappa * rho[(size_t)(y0 + q) * nx + gx];
        }
        SL[(r + 1) * BW + c + 1] = s;
    };
    lbar(tx, ty);
    for (int h = tid; h < halo_count<1>(th); h += tn) {
        int c, r;
        halo_point<1>(th, h, c, r);
        if (!g.walls || y0 + r <= ny - 1) lbar(c, r);
    }
    __syncthreads();
    if (!node) return;

    const int ka = (ty + 2) * AW + tx + 2;
    // div A: phibar of this node (and of the wall ghost folded onto it)
    const T pb = (dx12(nb_of<AW>(SX, tx + 2, ty + 2)) + dy12(nb_of<AW>(SY, tx + 2, ty + 2))) * T(1.0 / 12.0);
    T eb = pb * dphi + lap6(nb_of<BW>(SL, tx + 1, ty + 1)) * T(1.0 / 6.0);
    // the column's: its own point and the one beyond it
    const bool edge = g.bc_x && (x == 1 || x == nx - 2);
    const int side_x = x == 1 ? 0 : 1, xb = side_x ? nx - 1 : 0;
    const T sgx = side_x ? T(-1) : T(1);
    T cbar = 0, dphi_c = 0;
    if (edge) {
        const size_t cb = (size_t)y * nx + xb;
        const int kl = (ty + 1) * BW + tx + 1, d = side_x ? 1 : -1;
        const T lc = SL[kl + d], lv = SL[kl + d + BW] + SL[kl + d - BW];
        const T li = SL[kl], lvi = SL[kl + BW] + SL[kl - BW];
        dphi_c = fld[F_DPHI * N + cb];
        const T pc = (sgx * (T(4) * SX[ka] + SX[ka + AW] + SX[ka - AW]) + (SY[ka + AW] - SY[ka - AW])) * T(1.0 / 12.0);
        cbar = R[cb] + pc * dphi_c + ((T(4) * (li + lv) + lvi - T(20) * lc) + (T(4) * lc + lv)) * T(1.0 / 6.0);
    }
    if (g.walls && (y <= 2 || y >= ny - 3)) {
        for (int side = 0; side < 2; ++side) {
            const int dist = side ? ny - 2 - y : y - 1;  // rows from the wall row
            const T sg = side ? T(-1) : T(1);
            if (dist > 1) continue;
            // -div C, C at the wall row only (and its mirror image)
            const T *Cx = Cw + 2 * side * nx, *Cy = Cx + nx;
            auto cv = [&](const T *p, int xx) {
                if (g.bc_x) return xx >= 1 && xx <= nx - 2 ? p[xx] : T(0);
                return p[pmod(xx, nx)];
            };
            const T d = cv(Cx, x + 1) - cv(Cx, x - 1), s = T(4) * cv(Cy, x) + cv(Cy, x + 1) + cv(Cy, x - 1);
            eb -= (dist == 0 ? T(5) * d + sg * s : d - sg * s) * T(1.0 / 12.0);
            if (edge) {
                const T dc = sgx * cv(Cx, x), sc = cv(Cy, x);
                cbar -= (dist == 0 ? T(5) * dc + sg * sc : dc - sg * sc) * T(1.0 / 12.0);
            }
            if (dist == 0 && g.wet != T(0)) {
                // phibar of the ghost point, weighted at the shifted density
                const T pg = ((SX[ka + 1] - SX[ka - 1]) + sg * (T(4) * SY[ka] + SY[ka + 1] + SY[ka - 1])) * T(1.0 / 12.0);
                eb += pg * ((g.k2 * cs_dp0(g, rho[cn] + g.wet) - T(1.0 / 3.0)) - dphi);
                if (edge) {
                    const T pgc = (sgx * SX[ka] + sg * SY[ka]) * T(1.0 / 12.0);
                    cbar += pgc * ((g.k2 * cs_dp0(g, rho[(size_t)y * nx + xb] + g.wet) - T(1.0 / 3.0)) - dphi_c);
                }
            }
        }
    }
    rb += eb;
    if (edge) {
        T dth;
        const T th = col_theta(g, rho[cn], dth);
        const T gg = side_x ? g.g_out : g.g_in, ll = side_x ? g.l_out : g.l_in;
        rb += cbar * dth * (ll - gg);
        colp[(side_x * ny + y) * 2 + 0] += (double)(cbar * (T(1) - th));
        colp[(side_x * ny + y) * 2 + 1] += (double)(cbar * th);
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        T v = rb;
        acc_c(v, ex_(i), jx);
        acc_c(v, ey_(i), jy);
        lam_out[i * N + cn] = PART ? lam_out[i * N + cn] + v : v;
    }
}

// The same for channels between walls and pressure columns in FP32 (1024 x 256:
// three kernels of 26 us together became this one), the terms of
// every sum added one by one: Lbar and phibar on the ring around the tile,
// Ebar at this node's points of the ghost-extended lattice (itself, its mirror
// images behind the walls), then their sum. Only for tile heights that keep the
// two rows next to a wall in one tile (rows % th != 1), whose ring then holds all
// of it: beyond the ghost row or the column Lbar is zero.
template <bool PART>
__global__ void __launch_bounds__(TX * TMAX) adj_finish_terms(AdjGeo<float> g, int th, const float *__restrict__ fld,
                                                              const float *Ax, const float *Ay, const float *Jbx,
                                                              const float *Jby, const float *R, const float *Cw,
                                                              float *lam_out, double *colp)
{
    using T = float;
    __shared__ T SX[SMEM_A], SY[SMEM_A], SR[SMEM_A], SL[SMEM_B], SP[SMEM_B];
    chain_start();
    const int tid = threadIdx.x, tx = tid & (TX - 1), ty = tid / TX, tn = TX * th;
    const int nx = g.nx, ny = g.ny, ntx = (nx + TX - 1) / TX, by = blockIdx.x / ntx;
    const int x0 = (blockIdx.x - by * ntx) * TX, y0 = 1 + by * th;
    const int x = x0 + tx, y = y0 + ty;
    const size_t N = (size_t)nx * ny;
    const T *rho = fld + F_RHO * N;

    // Fbar (zero outside the fluid) and rho on the tile and two nodes around it
    auto load = [&](int c, int r) {
        const int gx = x0 + c, gy = y0 + r;
        T ax = 0, ay = 0, rv = 0;
        if (gx >= 1 && gx <= nx - 2 && gy >= 1 && gy <= ny - 2) {
            const size_t q = (size_t)gy * nx + gx;
            ax = Ax[q];
            ay = Ay[q];
            rv = rho[q];
        }
        const int k = (r + 2) * AW + c + 2;
        SX[k] = ax;
        SY[k] = ay;
        SR[k] = rv;
    };
    load(tx, ty);
    for (int h = tid; h < halo_count<2>(th); h += tn) {
        int c, r;
        halo_point<2>(th, h, c, r);
        load(c, r);
    }
    const bool node = x >= 1 && x <= nx - 2 && y <= ny - 2;
    const size_t cn = (size_t)y * nx + x;
    T rl = 0, jx = 0, jy = 0;
    if (node) {
        rl = R[cn];
        jx = Jbx[cn];
        jy = Jby[cn];
    }
    __syncthreads();

    auto bars = [&](int c, int r) {
        const int gx = x0 + c, gy = y0 + r, k = (r + 2) * AW + c + 2;
        T lb = 0, pb = 0;
        if ((gy == 1 || gy == ny - 2) && gx >= 1 && gx <= nx - 2) lb = -g.w_p * g.kappa * SR[k];
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            const int q = k - ey_(i) * AW - ex_(i);
            T s = 0;
            if (ex_(i) != 0) s += T(ex_(i)) * SX[q];
            if (ey_(i) != 0) s += T(ey_(i)) * SY[q];
            s *= T(3) * wq<T>(i);
            lb += g.kappa * SR[q] * s;
            pb -= s;
        }
        SL[(r + 1) * BW + c + 1] = lb;
        SP[(r + 1) * BW + c + 1] = pb;
    };
    bars(tx, ty);
    for (int h = tid; h < halo_count<1>(th); h += tn) {
        int c, r;
        halo_point<1>(th, h, c, r);
        bars(c, r);
    }
    __syncthreads();
    if (!node) return;

    // Lbar / phibar at an extended point; zero beyond the ring
    auto at = [&](const T *S, int px, int py) {
        const int c = px - x0 + 1, r = py - y0 + 1;
        return c >= 0 && c < BW && r >= 0 && r < th + 2 ? S[r * BW + c] : T(0);
    };
    // the point's own part; here and below, which products are fused is fixed,
    // since the compiler's choice differs between branches
    auto own = [](T pb, T dp, T lb) {
        return __fmaf_rn(-(T(6) * (T(1) - wq<T>(0))), lb, __fmul_rn(pb, dp));
    };
    // Ebar at the extended point (px, py), whose density has dphi = dp
    auto ebar = [&](int px, int py, T dp) {
        T eb = 0;
        if (px >= -1 && px <= nx && py >= -1 && py <= ny) {
            eb = own(at(SP, px, py), dp, at(SL, px, py));
        }
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            const int qx = px - ex_(i), qy = py - ey_(i);
            if ((qy == 1 || qy == ny - 2) && qx >= 1 && qx <= nx - 2) {
                const T *C = Cw + (qy == 1 ? 0 : 2 * nx) + qx;
                T s = 0;
                if (ex_(i) != 0) s += T(ex_(i)) * C[0];
                if (ey_(i) != 0) s += T(ey_(i)) * C[nx];
                eb = __fmaf_rn(T(3) * wq<T>(i), s, eb);
            }
            if (qx >= -1 && qx <= nx && qy >= -1 && qy <= ny) eb = __fmaf_rn(T(6) * wq<T>(i), at(SL, qx, qy), eb);
        }
        return eb;
    };
    const T *dphi = fld + F_DPHI * N;
    // dphi at the extended point (px, py), an image of lattice node (mx, y)
    auto dphi_at = [&](int mx, int py) {
        const T d = dphi[(size_t)y * nx + mx];
        if ((py > 0 && py < ny - 1) || g.wet == T(0)) return d;
        return g.k2 * cs_dp0(g, rho[(size_t)y * nx + mx] + g.wet) - T(1) / T(3);
    };
    // the extended rows whose density is this row's: itself, its mirror images
    T s = 0;
    const int v[3] = {y, 1 - y, 2 * ny - 3 - y};
    const bool low = y <= 2, high = y >= ny - 3;
    if (low || high) {
        s += ebar(x, v[0], dphi[cn]);
        if (low) s += ebar(x, v[1], dphi_at(x, v[1]));
        if (high) s += ebar(x, v[2], dphi_at(x, v[2]));
    } else {
        // away from the walls: no objective source, every neighbour on the ring
        const T *l = SL + (ty + 1) * BW + tx + 1;
        s = own(SP[(ty + 1) * BW + tx + 1], dphi[cn], l[0]);
#pragma unroll
        for (int i = 1; i < 9; ++i) s = __fmaf_rn(T(6) * wq<T>(i), l[-ey_(i) * BW - ex_(i)], s);
    }
    T rb = rl + s;
    if (x == 1 || x == nx - 2) {
        const int side = x == 1 ? 0 : 1, xb = side ? nx - 1 : 0, d = side ? 1 : -1;
        T t = 0;
        for (int m = 0; m < 3; ++m) {
            if ((m == 1 && !low) || (m == 2 && !high)) continue;
            const T dp = dphi_at(xb, v[m]);
            t += ebar(xb, v[m], dp);
            t += ebar(xb + d, v[m], dp);
        }
        const T rbb = R[(size_t)y * nx + xb] + t;
        T dth;
        const T w = col_theta(g, rho[cn], dth);
        const T gg = side ? g.g_out : g.g_in, ll = side ? g.l_out : g.l_in;
        rb += rbb * dth * (ll - gg);
        colp[(side * ny + y) * 2 + 0] += (double)(rbb * (T(1) - w));
        colp[(side * ny + y) * 2 + 1] += (double)(rbb * w);
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        T u = rb;
        acc_c(u, ex_(i), jx);
        acc_c(u, ey_(i), jy);
        lam_out[i * N + cn] = PART ? lam_out[i * N + cn] + u : u;
    }
}

// One-block deterministic sums: acc[slot + k] += sum over the k-th series.
constexpr int RED_THREADS = 512;
__global__ void adj_reduce(const double *__restrict__ a, long long stride_a, long long len, int nseries,
                           double *acc)
{
    __shared__ double sh[RED_THREADS];
    for (int k = 0; k < nseries; ++k) {
        double s = 0.0;
        for (long long i = threadIdx.x; i < len; i += RED_THREADS) s += a[k * stride_a + i];
        sh[threadIdx.x] = s;
        __syncthreads();
        for (int h = RED_THREADS / 2; h > 0; h >>= 1) {
            if ((int)threadIdx.x < h) sh[threadIdx.x] += sh[threadIdx.x + h];
            __syncthreads();
        }
        if (threadIdx.x == 0) acc[k] += sh[0];
        __syncthreads();
    }
}

// colp holds (side, row, {gas, liquid}) pairs; sums into acc[0..3] as
// (gas_in, liq_in, gas_out, liq_out).
__global__ void adj_reduce_col(const double *__restrict__ colp, int ny, double *acc)
{
    __shared__ double sh[RED_THREADS];
    for (int k = 0; k < 4; ++k) {
        const int side = k / 2, br = k % 2;
        double s = 0.0;
        for (int y = threadIdx.x; y < ny; y += RED_THREADS) s += colp[(side * ny + y) * 2 + br];
        sh[threadIdx.x] = s;
        __syncthreads();
        for (int h = RED_THREADS / 2; h > 0; h >>= 1) {
            if ((int)threadIdx.x < h) sh[threadIdx.x] += sh[threadIdx.x + h];
            __syncthreads();
        }
        if (threadIdx.x == 0) acc[k] += sh[0];
        __syncthreads();
    }
}

// the resting equilibrium of rho0, in the state layout (padding columns stay as set)
template <typename S>
__global__ void adj_init_f(AdjGeo<double> g, const double *__restrict__ rho0, S *f)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= g.nx * g.ny) return;
    const int x = c % g.nx, y = c / g.nx;
    for (int i = 0; i < 9; ++i) f[((size_t)y * 9 + i) * g.fp + x] = (S)(wq<double>(i) * rho0[c]);
}

template <typename T>
__global__ void adj_grad_rho0(const T *__restrict__ lam, int n, double *g)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    double s = 0.0;
    for (int i = 0; i < 9; ++i) s += wq<double>(i) * (double)lam[i * n + c];
    g[c] = s;
}

constexpr int TPB = 256;
inline unsigned blocks(long long m) { return (unsigned)((m + TPB - 1) / TPB); }

// Fields of the states of a block are computed for as many states at once as
// fit this many bytes (at least one): enough to fill the GPU from a small
// lattice, bounded on a large one. Two such buffers are kept.
constexpr size_t FIELD_BYTES = (size_t)256 << 20;

} // namespace

struct lbm_adjoint {
    lbm_grid grid{};
    lbm_eos eos{};
    lbm_drive drive{};
    double tau = 1, wet = 0;
    int64_t nsteps = 0, K = 0, nblocks = 0;
    cudaStream_t stream = nullptr;
    lbm_ctx *ctx = nullptr;
    bool have_drive = false, forward_done = false;
    lbm_collision coll{};  // BGK unless set
    AdjGeo<double> geo{};
    int rprec = 64;  // reverse sweep (and objective) arithmetic: 64 or 32
    double dgin = 0, dlin = 0, dgout = 0, dlout = 0;  // d rho_column / d dp
    int64_t held = -1;  // block whose recomputed states blk holds (-1: none)
    int64_t G = 1;      // states whose fields one buffer of fld holds
    // The backward pass recomputes states and their fields on `prep` while the
    // reverse chain runs on `chain`, from the other of two field buffers (one
    // buffer and the caller's stream alone where memory is short).
    bool overlap = false;
    cudaStream_t chain = nullptr, prep = nullptr;
    cudaEvent_t ev_begin = nullptr, ev_end = nullptr, ev_fld[2] = {nullptr, nullptr}, ev_chain[2] = {nullptr, nullptr};
    int sms = 1;
    // device buffers (the reverse sweep's fields and adjoint populations are
    // sized for doubles and hold floats with rprec = 32)
    double *ckpt = nullptr, *blk = nullptr, *lam0 = nullptr, *lam1 = nullptr, *fld[2] = {nullptr, nullptr};
    double *Ax = nullptr, *Ay = nullptr, *Jbx = nullptr, *Jby = nullptr, *R = nullptr, *Cw = nullptr;
    double *loads = nullptr, *tw = nullptr, *colp = nullptr, *acc = nullptr, *rho0 = nullptr, *AS = nullptr;
    std::vector<void *> allocs;
    std::string err;
};

namespace {

lbm_status adj_fail(lbm_adjoint *a, cudaError_t e, const char *what)
{
    a->err = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA;
}

#define ACK(expr, what)                              \
    do {                                             \
        cudaError_t e_ = (expr);                     \
        if (e_ != cudaSuccess) return adj_fail(a, e_, what); \
    } while (0)

lbm_status adj_alloc(lbm_adjoint *a, double **p, size_t count)
{
    void *q = nullptr;
    ACK(cudaMalloc(&q, count * sizeof(double)), "adjoint allocation");
    a->allocs.push_back(q);
    *p = (double *)q;
    return LBM_OK;
}

size_t npop(const lbm_adjoint *a) { return (size_t)9 * a->grid.nx * a->grid.ny; }
// one stored state in the forward context's own layout (plane pitch pitch_of(nx))
size_t spop(const lbm_adjoint *a) { return (size_t)9 * lbm::pitch_of(a->grid.nx) * a->grid.ny; }
// bytes of one stored state (the forward precision, padded to 256 bytes: the
// step's bulk and tensor copies read it in place), and state k of an array of them
size_t sbytes(const lbm_adjoint *a)
{
    return (spop(a) * (a->grid.precision == 32 ? 4 : 8) + 255) / 256 * 256;
}
void *state_at(double *base, size_t k, size_t bytes) { return (char *)base + k * bytes; }
// state t of the trajectory: a checkpoint, or its place in the block
void *state_of(lbm_adjoint *a, int64_t t)
{
    const size_t SB = sbytes(a);
    return t % a->K == 0 ? state_at(a->ckpt, (size_t)(t / a->K), SB) : state_at(a->blk, (size_t)(t % a->K), SB);
}
States block_states(lbm_adjoint *a, int64_t b)
{
    return States{(const char *)state_at(a->ckpt, (size_t)b, sbytes(a)), (const char *)a->blk, sbytes(a)};
}

template <typename T>
T *as(double *p) { return reinterpret_cast<T *>(p); }

// Launch with programmatic stream serialization (`chained`): the kernel's launch
// overlaps the previous kernel of the chain, which it waits for before any access.
template <typename... P, typename... Q>
cudaError_t launch_chained(void (*k)(P...), dim3 grid, dim3 block, cudaStream_t st, bool chained, Q &&...q)
{
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, static_cast<P>(q)...);
}

unsigned tiles(int len, int t) { return (unsigned)((len + t - 1) / t); }
int fluid_rows(const AdjGeo<double> &g) { return g.walls ? g.ny - 2 : g.ny; }

// the wall loads of the states of block b (n of them), added to the sums
template <typename T>
lbm_status adj_objective_t(lbm_adjoint *a, int64_t b, int n)
{
    const AdjGeo<T> g = geo_as<T>(a->geo);
    const States st = block_states(a, b);
    for (int m = 0; m < n; m += (int)a->G) {
        const int c = (int)std::min<int64_t>(a->G, n - m);
        const dim3 grid(tiles(g.nx, LT), 2, c);
        if (a->grid.precision == 32) adj_loads<float, T><<<grid, 128, 0, a->stream>>>(g, st, m, a->loads);
        else adj_loads<double, T><<<grid, 128, 0, a->stream>>>(g, st, m, a->loads);
        adj_add_loads<<<blocks(4LL * g.nx), TPB, 0, a->stream>>>(a->loads, 4 * g.nx, c, a->tw);
    }
    ACK(cudaGetLastError(), "adjoint objective kernels");
    return LBM_OK;
}

lbm_status adj_objective(lbm_adjoint *a, int64_t b, int n)
{
    if (!a->geo.walls) return LBM_OK;  // no wall loads
    return a->rprec == 32 ? adj_objective_t<float>(a, b, n) : adj_objective_t<double>(a, b, n);
}

// Tile height for `states` lattices stepped by one launch: the one whose
// busiest SM has the least rows to do (a tile costs its rows and about two
// more for its halo).
int tile_rows(const lbm_adjoint *a, int states)
{
    const long long ntx = tiles(a->geo.nx, TX), rows = fluid_rows(a->geo);
    int best = 8;
    long long least = -1;
    for (int th = 4; th <= TMAX; ++th) {
        if (rows % th == 1) continue;  // adj_finish_terms: the two rows next to a wall share a tile (adj_chain_t)
        const long long t = ntx * ((rows + th - 1) / th) * states, cost = (t + a->sms - 1) / a->sms * (th + 2);
        if (least < 0 || cost < least) { least = cost; best = th; }
    }
    return best;
}

// A run of states m0 .. m1-1 of block b, walked in reverse from one field buffer.
struct Run {
    int64_t b;
    int m0, m1;
};

// the fields of a run's states into buffer `buf`, on `st`
template <typename T>
lbm_status adj_fields_t(lbm_adjoint *a, const Run &r, int buf, cudaStream_t st)
{
    const AdjGeo<T> g = geo_as<T>(a->geo);
    const States states = block_states(a, r.b);
    const size_t N = (size_t)g.nx * g.ny;
    const int n = r.m1 - r.m0, fh = tile_rows(a, n);
    const dim3 ng((unsigned)((N + 127) / 128), n), fg(tiles(g.nx, TX) * tiles(fluid_rows(a->geo), fh), n);
    T *f = as<T>(a->fld[buf]);
    if (a->grid.precision == 32) adj_nodes<float, T><<<ng, 128, 0, st>>>(g, states, r.m0, f);
    else adj_nodes<double, T><<<ng, 128, 0, st>>>(g, states, r.m0, f);
    adj_forces<T><<<fg, TX * fh, 0, st>>>(g, fh, f);
    ACK(cudaGetLastError(), "adjoint field kernels");
    return LBM_OK;
}

// reverse steps over a run's states, last first; lin / lout swap per step
template <typename T, bool PART>
lbm_status adj_chain_t(lbm_adjoint *a, const Run &r, int buf, cudaStream_t st, double *&lin, double *&lout)
{
    const AdjGeo<T> g = geo_as<T>(a->geo);
    const size_t N = (size_t)g.nx * g.ny;
    constexpr int LB = sizeof(T) == 8 ? 64 : 128;
    const unsigned eblocks = g.bc_x ? tiles(2 * g.ny, LB) : 0, nblocks = eblocks + (unsigned)((N + LB - 1) / LB);
    const int th = tile_rows(a, 1);
    const unsigned tg = tiles(g.nx, TX) * tiles(fluid_rows(a->geo), th);
    for (int m = r.m1 - 1; m >= r.m0; --m) {
        const T *f = as<T>(a->fld[buf]) + (size_t)(m - r.m0) * NFIELD * N;
        T *li = as<T>(lin), *lo = as<T>(lout);
        // a run's first kernel is launched plainly: its fields were written by
        // the kernels or events before it in the stream
        ACK(launch_chained(adj_local<T, PART, LB>, dim3(nblocks), dim3(LB), st, m + 1 < r.m1, g, (int)eblocks, li, f, lo,
                           as<T>(a->Ax), as<T>(a->Ay), as<T>(a->Jbx), as<T>(a->Jby), as<T>(a->R), as<T>(a->Cw), a->AS),
            "adjoint local kernel");
        auto finish = adj_finish<T, PART>;
        if constexpr (BY_TERMS<T>) {
            // where every height leaves a single row (rows = 1 mod 720720): adj_finish
            if (g.walls && g.bc_x && (g.ny - 2) % th != 1) finish = adj_finish_terms<PART>;
        }
        ACK(launch_chained(finish, dim3(tg), dim3(TX * th), st, true, g, th, f, as<T>(a->Ax), as<T>(a->Ay), as<T>(a->Jbx),
                           as<T>(a->Jby), as<T>(a->R), as<T>(a->Cw), lo, a->colp),
            "adjoint finish kernel");
        std::swap(lin, lout);
    }
    return LBM_OK;
}

lbm_status adj_run_fields(lbm_adjoint *a, const Run &r, int buf, cudaStream_t st)
{
    return a->rprec == 32 ? adj_fields_t<float>(a, r, buf, st) : adj_fields_t<double>(a, r, buf, st);
}
lbm_status adj_run_chain(lbm_adjoint *a, const Run &r, int buf, cudaStream_t st, double *&lin, double *&lout)
{
    // without MRT and at tau = 1 the relaxation leaves nothing of f*-bar
    const bool part = a->geo.mrt || a->geo.inv_tau != 1.0;
    if (a->rprec == 32)
        return part ? adj_chain_t<float, true>(a, r, buf, st, lin, lout)
                    : adj_chain_t<float, false>(a, r, buf, st, lin, lout);
    return part ? adj_chain_t<double, true>(a, r, buf, st, lin, lout)
                : adj_chain_t<double, false>(a, r, buf, st, lin, lout);
}

// The whole reverse sweep: block by block, last first, each in runs of at most G
// states. Preparing run i + 1 (recomputing its block's states first, where it
// opens one: by then the fields of every state in their storage are taken)
// does not depend on the adjoint, so it overlaps the chain of run i, whose two
// short kernels per step leave most of the FP64 pipe idle (512 x 128, 200 steps
// forward and back: 14.1 ms one after the other, 11.4 overlapped; 1024 x 256
// with an FP32 reverse, 100 steps: 6.2 and 5.7). Run i's fields lie in buffer
// i & 1, free again once chain i - 2 is through.
lbm_status adj_sweep(lbm_adjoint *a, double *&lin, double *&lout)
{
    std::vector<Run> runs;
    for (int64_t b = a->nblocks - 1; b >= 0; --b) {
        const int n = (int)(std::min(a->nsteps, (b + 1) * a->K) - b * a->K);
        const int parts = (int)((n + a->G - 1) / a->G), len = (n + parts - 1) / parts;
        for (int m1 = n; m1 > 0; m1 -= len) runs.push_back(Run{b, std::max(0, m1 - len), m1});
    }
    const bool ov = a->overlap;
    const cudaStream_t prep = ov ? a->prep : a->stream, chain = ov ? a->chain : a->stream;
    lbm_status s;
    auto prepare = [&](size_t i) -> lbm_status {
        const Run &r = runs[i];
        if (a->held != r.b) {
            a->held = -1;
            const int64_t n0 = r.b * a->K, n1 = std::min(a->nsteps, n0 + a->K);
            for (int64_t t = n0; t + 1 < n1; ++t)
                ACK(lbm_ctx_step_between(a->ctx, state_of(a, t), state_of(a, t + 1), prep), "recompute step");
            a->held = r.b;
        }
        const int buf = ov ? (int)(i & 1) : 0;
        if (ov && i >= 2) ACK(cudaStreamWaitEvent(prep, a->ev_chain[buf], 0), "adjoint event");
        if ((s = adj_run_fields(a, r, buf, prep)) != LBM_OK) return s;
        if (ov) ACK(cudaEventRecord(a->ev_fld[buf], prep), "adjoint event");
        return LBM_OK;
    };
    if (ov) {
        ACK(cudaEventRecord(a->ev_begin, a->stream), "adjoint event");
        ACK(cudaStreamWaitEvent(prep, a->ev_begin, 0), "adjoint event");
        ACK(cudaStreamWaitEvent(chain, a->ev_begin, 0), "adjoint event");
        if ((s = prepare(0)) != LBM_OK) return s;
    }
    for (size_t i = 0; i < runs.size(); ++i) {
        const int buf = ov ? (int)(i & 1) : 0;
        if (!ov) {
            if ((s = prepare(i)) != LBM_OK) return s;
        } else {
            if (i + 1 < runs.size() && (s = prepare(i + 1)) != LBM_OK) return s;
            ACK(cudaStreamWaitEvent(chain, a->ev_fld[buf], 0), "adjoint event");
        }
        if ((s = adj_run_chain(a, runs[i], buf, chain, lin, lout)) != LBM_OK) return s;
        if (ov) ACK(cudaEventRecord(a->ev_chain[buf], chain), "adjoint event");
    }
    if (ov) {  // every event of `prep` was waited for on `chain`
        ACK(cudaEventRecord(a->ev_end, chain), "adjoint event");
        ACK(cudaStreamWaitEvent(a->stream, a->ev_end, 0), "adjoint event");
    }
    return LBM_OK;
}

// Work left on the internal streams by a call that failed half way is finished
// before anything new is enqueued.
cudaError_t adj_drain(lbm_adjoint *a)
{
    if (!a->overlap) return cudaSuccess;
    cudaError_t e = cudaStreamSynchronize(a->prep);
    return e == cudaSuccess ? cudaStreamSynchronize(a->chain) : e;
}

// the error word of the forward context's steps, read with the results
lbm_status step_errors(lbm_adjoint *a, int word, const char *what)
{
    if (!word) return LBM_OK;
    const lbm_status s = word & 1 ? LBM_ERR_NAN : LBM_ERR_TIMEOUT;
    a->err = std::string(what) + ": " + lbm_status_string(s);
    return s;
}

// the sweep's internal streams and events; false (nothing kept) on failure.
// The chain, whose kernels are short and wait for one another, goes first
// where both have blocks to place.
void adj_streams_free(lbm_adjoint *a)
{
    for (cudaEvent_t *e : {&a->ev_begin, &a->ev_end, &a->ev_fld[0], &a->ev_fld[1], &a->ev_chain[0], &a->ev_chain[1]}) {
        if (*e) cudaEventDestroy(*e);
        *e = nullptr;
    }
    for (cudaStream_t *st : {&a->chain, &a->prep}) {
        if (*st) cudaStreamDestroy(*st);
        *st = nullptr;
    }
}
bool adj_streams(lbm_adjoint *a)
{
    int least = 0, greatest = 0;
    cudaError_t e = cudaDeviceGetStreamPriorityRange(&least, &greatest);
    if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&a->chain, cudaStreamNonBlocking, greatest);
    if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&a->prep, cudaStreamNonBlocking, least);
    for (cudaEvent_t *ev : {&a->ev_begin, &a->ev_end, &a->ev_fld[0], &a->ev_fld[1], &a->ev_chain[0], &a->ev_chain[1]})
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
    if (e == cudaSuccess) return true;
    adj_streams_free(a);
    return false;
}

lbm_status ctx_status(lbm_adjoint *a, lbm_status s, const char *what)
{
    if (s != LBM_OK) {
        const char *m = a->ctx ? lbm_last_error(a->ctx) : "";
        a->err = std::string(what) + ": " + lbm_status_string(s) + (m && *m ? std::string(" (") + m + ")" : "");
    }
    return s;
}

bool same_drive(const lbm_drive &x, const lbm_drive &y)
{
    auto eq = [](double u, double v) { return u == v || (std::isnan(u) && std::isnan(v)); };
    return eq(x.dp, y.dp) && eq(x.p_ref, y.p_ref) && eq(x.gx, y.gx) && eq(x.gy, y.gy);
}

// (Re)build the FP64 forward context for a drive and the adjoint's geometry.
lbm_status adj_setup_drive(lbm_adjoint *a, const lbm_drive *drive)
{
    lbm_drive d = drive ? *drive : lbm_drive{0.0, NAN, 0.0, 0.0};
    if (a->ctx && a->have_drive && same_drive(d, a->drive)) return LBM_OK;
    if (a->ctx) { lbm_free(a->ctx); a->ctx = nullptr; }
    std::vector<double> one((size_t)a->grid.nx * a->grid.ny, 0.1);
    lbm_status s = lbm_init(&a->grid, &a->eos, a->tau, nullptr, a->wet, &d, one.data(), nullptr, 0, a->stream, &a->ctx);
    if (s != LBM_OK) { a->err = std::string("forward context: ") + lbm_status_string(s); a->ctx = nullptr; return s; }
    if ((s = lbm_set_collision(a->ctx, &a->coll)) != LBM_OK) return ctx_status(a, s, "collision");
    a->drive = d;
    a->have_drive = true;
    lbm_diag_t dg;
    s = lbm_diag(a->ctx, &dg);
    if (s != LBM_OK) return ctx_status(a, s, "forward context diag");

    AdjGeo<double> &g = a->geo;
    g.nx = a->grid.nx; g.ny = a->grid.ny; g.walls = a->grid.walls; g.bc_x = a->grid.bc_x;
    g.fp = lbm::pitch_of(a->grid.nx);
    lbm::Thermo th{};
    double tc;
    if (lbm::thermo_of(a->eos, &th, &tc)) { a->err = "equation of state"; return LBM_ERR_PARAM; }
    g.eos_kind = th.kind; g.bpr = th.b; g.aalpha = th.aalpha;
    g.RT = a->eos.R * dg.T; g.a = a->eos.a; g.b4 = 0.25 * a->eos.b; g.k2 = a->eos.k * a->eos.k;
    g.kappa = a->eos.kappa; g.tau = a->tau; g.inv_tau = 1.0 / a->tau; g.nu = (a->tau - 0.5) / 3.0; g.wet = a->wet;
    g.mrt = a->coll.kind == LBM_COLL_MRT;
    g.ushift = g.mrt ? 1.0 / a->coll.s_j : a->tau;
    if (g.mrt) {
        const double s_nu = a->coll.s_nu > 0 ? a->coll.s_nu : 1.0 / a->tau;
        const double r[9] = {0.0, a->coll.s_e / 36.0, a->coll.s_eps / 36.0, a->coll.s_j / 6.0, a->coll.s_q / 12.0,
                             a->coll.s_j / 6.0, a->coll.s_q / 12.0, s_nu / 4.0, s_nu / 4.0};
        for (int k = 0; k < 9; ++k) g.mrate[k] = r[k];
    }
    g.gx = d.gx; g.gy = d.gy;
    g.g_in = dg.rho_in; g.l_in = dg.rho_in_l; g.g_out = dg.rho_out; g.l_out = dg.rho_out_l;
    g.ph_g = dg.rho_g;
    g.inv_dph = dg.rho_l > dg.rho_g ? 1.0 / (dg.rho_l - dg.rho_g) : 0.0;
    // column densities are EOS roots of k^2 p0(rho) = p_ref +- dp/2, so
    // d rho / d dp = +-1 / (2 k^2 p0'(rho)); a density held at a spinodal
    // does not move with dp
    a->dgin = a->dlin = a->dgout = a->dlout = 0.0;
    if (a->grid.bc_x) {
        lbm::ChannelThermo ct;
        if (lbm::channel_thermo(a->eos, d, true, &ct)) { a->err = "column thermodynamics"; return LBM_ERR_PARAM; }
        auto rate = [&](double rho, bool sat, double sgn) {
            return sat ? 0.0 : sgn * 0.5 / (g.k2 * lbm::eos_dpressure(ct.th, rho));
        };
        a->dgin = rate(g.g_in, ct.sat[0], 1.0);
        a->dlin = rate(g.l_in, ct.sat[1], 1.0);
        a->dgout = rate(g.g_out, ct.sat[2], -1.0);
        a->dlout = rate(g.l_out, ct.sat[3], -1.0);
    }
    return LBM_OK;
}

} // namespace

extern "C" {

lbm_status lbm_adjoint_init(const lbm_grid *grid, const lbm_eos *eos, double tau, double wetting, int64_t nsteps,
                            int64_t block_steps, void *stream, lbm_adjoint **out)
{
    if (!out) return LBM_ERR_ARG;
    *out = nullptr;
    if (!grid || !eos || (grid->precision != 64 && grid->precision != 32) || nsteps < 1 || block_steps < 0)
        return LBM_ERR_ARG;
    if (grid->nx < 1 || grid->ny < 1 || 9ll * grid->nx * grid->ny >= (1ll << 31)) return LBM_ERR_ARG;
    if (!(tau > 0.5) || !std::isfinite(wetting)) return LBM_ERR_PARAM;
    lbm_adjoint *a = new (std::nothrow) lbm_adjoint();
    if (!a) return LBM_ERR_OOM;
    a->grid = *grid;
    a->eos = *eos;
    a->tau = tau;
    a->wet = wetting;
    a->nsteps = nsteps;
    a->K = block_steps > 0 ? block_steps : (int64_t)std::ceil(std::sqrt((double)nsteps));
    if (a->K > nsteps) a->K = nsteps;
    a->nblocks = (nsteps + a->K - 1) / a->K;
    a->stream = (cudaStream_t)stream;

    const size_t n = (size_t)grid->nx * grid->ny, P = npop(a);
    const size_t SD = sbytes(a) / 8;  // one stored state, in doubles
    a->G = (int64_t)std::min<size_t>(a->K, std::max<size_t>(1, FIELD_BYTES / (NFIELD * n * sizeof(double))));
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&a->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        lbm_adjoint_free(a);
        return LBM_ERR_CUDA;
    }
    a->G = std::min<int64_t>(a->G, 32768);  // states are a grid dimension of the field and load kernels
    lbm_status s = LBM_OK;
    struct { double **p; size_t count; } bufs[] = {
        {&a->ckpt, SD * a->nblocks}, {&a->blk, SD * a->K}, {&a->lam0, P}, {&a->lam1, P},
        {&a->Ax, n}, {&a->Ay, n}, {&a->Jbx, n}, {&a->Jby, n}, {&a->R, n}, {&a->Cw, 4 * (size_t)grid->nx},
        {&a->tw, 4 * (size_t)grid->nx}, {&a->colp, 4 * (size_t)grid->ny}, {&a->acc, 8}, {&a->rho0, n},
        {&a->AS, 2 * n}};
    for (auto &b : bufs)
        if (s == LBM_OK) s = adj_alloc(a, b.p, b.count);
    // Two field buffers and the overlapped sweep, or, where memory is short, the
    // fields of one state at a time on the caller's stream. The runs of a block
    // are of even length.
    const int64_t parts = (a->K + a->G - 1) / a->G;
    a->G = (a->K + parts - 1) / parts;
    const size_t F = NFIELD * n;
    if (s == LBM_OK) {
        double *two = nullptr;
        if (adj_alloc(a, &two, 2 * F * a->G + 4 * (size_t)grid->nx * a->G) == LBM_OK && adj_streams(a)) {
            a->fld[0] = two;
            a->fld[1] = two + F * a->G;
            a->loads = two + 2 * F * a->G;
            a->overlap = true;
        } else {
            cudaGetLastError();
            a->err.clear();
            a->G = 1;
            s = adj_alloc(a, &a->fld[0], F + 4 * (size_t)grid->nx);
            a->loads = a->fld[0] ? a->fld[0] + F : nullptr;
        }
    }
    if (s != LBM_OK) { lbm_adjoint_free(a); return s; }
    // slots that no population reaches and padding columns are never read as
    // lattice nodes; they start at zero once
    if (cudaMemsetAsync(a->ckpt, 0, SD * 8 * a->nblocks, a->stream) != cudaSuccess ||
        cudaMemsetAsync(a->blk, 0, SD * 8 * a->K, a->stream) != cudaSuccess) {
        lbm_adjoint_free(a);
        return LBM_ERR_CUDA;
    }
    // the forward context is built by the first forward, for its drive
    lbm::Thermo th{};
    double tc;
    if (lbm::thermo_of(*eos, &th, &tc)) { lbm_adjoint_free(a); return LBM_ERR_PARAM; }
    *out = a;
    return LBM_OK;
}

lbm_status lbm_adjoint_forward(lbm_adjoint *a, const lbm_drive *drive, const double *rho0, double *J)
{
    if (!a || !rho0 || !J) return LBM_ERR_ARG;
    a->forward_done = false;
    ACK(adj_drain(a), "adjoint streams");
    lbm_status s = adj_setup_drive(a, drive);
    if (s != LBM_OK) return s;
    const long long n = (long long)a->grid.nx * a->grid.ny;
    a->held = -1;
    ACK(cudaMemcpyAsync(a->rho0, rho0, n * sizeof(double), cudaMemcpyDefault, a->stream), "rho0 copy");
    if (a->grid.precision == 32)
        adj_init_f<float><<<blocks(n), TPB, 0, a->stream>>>(a->geo, a->rho0, (float *)a->ckpt);
    else
        adj_init_f<double><<<blocks(n), TPB, 0, a->stream>>>(a->geo, a->rho0, a->ckpt);
    ACK(cudaGetLastError(), "adjoint init kernel");
    int *ew = lbm_ctx_error_word(a->ctx);
    ACK(cudaMemsetAsync(ew, 0, sizeof(int), a->stream), "adjoint memset");
    ACK(cudaMemsetAsync(a->acc, 0, 8 * sizeof(double), a->stream), "adjoint memset");
    ACK(cudaMemsetAsync(a->tw, 0, 4 * (size_t)a->grid.nx * sizeof(double), a->stream), "adjoint memset");
    // Each step writes the next stored state in place (no copy); the wall loads
    // of a block's states are taken together once they are all there.
    for (int64_t t = 0; t < a->nsteps; ++t) {
        const bool last = t + 1 == a->nsteps;
        if (!last) ACK(lbm_ctx_step_between(a->ctx, state_of(a, t), state_of(a, t + 1), a->stream), "forward step");
        // the step that ends a block writes the next checkpoint, not the block
        if ((last || (t + 1) % a->K == 0) && (s = adj_objective(a, t / a->K, (int)(t % a->K) + 1)) != LBM_OK) return s;
    }
    // tw and pw are adjacent: two series of 2 nx per-column sums over the steps
    adj_reduce<<<1, RED_THREADS, 0, a->stream>>>(a->tw, 2LL * a->grid.nx, 2LL * a->grid.nx, 2, a->acc);
    ACK(cudaGetLastError(), "adjoint objective sum");
    double h[2];
    int word = 0;
    ACK(cudaMemcpyAsync(h, a->acc, 2 * sizeof(double), cudaMemcpyDeviceToHost, a->stream), "objective copy");
    ACK(cudaMemcpyAsync(&word, ew, sizeof(int), cudaMemcpyDeviceToHost, a->stream), "objective copy");
    ACK(cudaStreamSynchronize(a->stream), "forward sync");
    if ((s = step_errors(a, word, "forward step")) != LBM_OK) return s;
    J[0] = h[0];
    J[1] = h[1];
    a->held = a->nblocks - 1;  // the last block's states are still there
    a->forward_done = true;
    return LBM_OK;
}

lbm_status lbm_adjoint_backward(lbm_adjoint *a, double w_tau, double w_p, double *grad_rho0, double *grad_drive)
{
    if (!a || !grad_rho0 || !grad_drive) return LBM_ERR_ARG;
    if (!a->forward_done) { a->err = "backward before forward"; return LBM_ERR_STATE; }
    if (!std::isfinite(w_tau) || !std::isfinite(w_p)) return LBM_ERR_ARG;
    ACK(adj_drain(a), "adjoint streams");
    a->geo.w_tau = w_tau;
    a->geo.w_p = w_p;
    const long long n = (long long)a->grid.nx * a->grid.ny;
    const size_t P = npop(a);
    ACK(cudaMemsetAsync(a->acc, 0, 8 * sizeof(double), a->stream), "adjoint memset");
    // both: solid rows and pressure columns stay zero in either
    ACK(cudaMemsetAsync(a->lam0, 0, P * sizeof(double), a->stream), "adjoint memset");
    ACK(cudaMemsetAsync(a->lam1, 0, P * sizeof(double), a->stream), "adjoint memset");
    ACK(cudaMemsetAsync(a->AS, 0, 2 * (size_t)n * sizeof(double), a->stream), "adjoint memset");
    ACK(cudaMemsetAsync(a->colp, 0, 4 * (size_t)a->grid.ny * sizeof(double), a->stream), "adjoint memset");
    double *lin = a->lam1, *lout = a->lam0;
    lbm_status s;
    if ((s = adj_sweep(a, lin, lout)) != LBM_OK) return s;
    // per-node and per-row sums over the steps, reduced once
    adj_reduce_col<<<1, RED_THREADS, 0, a->stream>>>(a->colp, a->grid.ny, a->acc + 2);
    adj_reduce<<<1, RED_THREADS, 0, a->stream>>>(a->AS, n, n, 2, a->acc + 6);
    if (a->rprec == 32)
        adj_grad_rho0<float><<<blocks(n), TPB, 0, a->stream>>>((const float *)lin, (int)n, a->rho0);
    else
        adj_grad_rho0<double><<<blocks(n), TPB, 0, a->stream>>>(lin, (int)n, a->rho0);
    ACK(cudaGetLastError(), "gradient kernel");
    ACK(cudaMemcpyAsync(grad_rho0, a->rho0, n * sizeof(double), cudaMemcpyDefault, a->stream), "gradient copy");
    double h[8];
    int word = 0;
    ACK(cudaMemcpyAsync(h, a->acc, 8 * sizeof(double), cudaMemcpyDeviceToHost, a->stream), "gradient copy");
    ACK(cudaMemcpyAsync(&word, lbm_ctx_error_word(a->ctx), sizeof(int), cudaMemcpyDeviceToHost, a->stream),
        "gradient copy");
    ACK(cudaStreamSynchronize(a->stream), "backward sync");
    if ((s = step_errors(a, word, "recompute step")) != LBM_OK) return s;
    // h[2..5]: sensitivities to the column densities (gas_in, liq_in, gas_out, liq_out)
    grad_drive[0] = h[2] * a->dgin + h[3] * a->dlin + h[4] * a->dgout + h[5] * a->dlout;
    grad_drive[1] = h[6];
    grad_drive[2] = h[7];
    return LBM_OK;
}

lbm_status lbm_adjoint_set_collision(lbm_adjoint *a, const lbm_collision *c)
{
    if (!a) return LBM_ERR_ARG;
    const lbm_collision prev = a->coll;
    a->coll = c ? *c : lbm_collision{};
    if (a->ctx) {
        lbm_status s = lbm_set_collision(a->ctx, &a->coll);
        if (s != LBM_OK) { a->coll = prev; return s; }
    } else if (a->coll.kind == LBM_COLL_MRT) {
        for (double r : {a->coll.s_e, a->coll.s_eps, a->coll.s_j, a->coll.s_q})
            if (!(r > 0.0 && r < 2.0)) { a->coll = prev; return LBM_ERR_ARG; }
    } else if (a->coll.kind != LBM_COLL_BGK) {
        a->coll = prev;
        return LBM_ERR_ARG;
    }
    a->have_drive = false;    // rebuild the geometry with the new collision
    a->forward_done = false;  // earlier checkpoints belong to the old operator
    return LBM_OK;
}

lbm_status lbm_adjoint_set_precision(lbm_adjoint *a, int32_t reverse_precision)
{
    if (!a || (reverse_precision != 32 && reverse_precision != 64)) return LBM_ERR_ARG;
    a->rprec = reverse_precision;
    return LBM_OK;
}

const char *lbm_adjoint_last_error(const lbm_adjoint *a) { return a ? a->err.c_str() : ""; }

void lbm_adjoint_free(lbm_adjoint *a)
{
    if (!a) return;
    adj_drain(a);
    if (a->ctx) lbm_free(a->ctx);
    adj_streams_free(a);
    for (void *p : a->allocs) cudaFree(p);
    delete a;
}

} // extern "C"
