// The FP64 step, the FP32 step of small grids, and the fields in either precision,
// by tiles of 32 columns by th rows, one node per thread.
//
// GB300 runs FP64 at 1/64 of the FP32 rate (two thread-instructions per clock
// and SM), so an FP64 step is bound by each SM's FP64 pipe: what counts is the
// number of FP64 instructions per node, that the pipe of every SM has work all
// the time, and that the SMs finish together. The strip kernel
// (lbm_kernels.cuh) holds 90 KB of stage and rings per CTA: two CTAs of four
// warps per SM, a barrier per row, 82% of the pipe on busy SMs and SMs busy 90%
// of the step; and a small grid gives it few CTAs (128 x 128: 64, each a serial
// chain of seven rows). Here a CTA needs only the densities, phi and Laplacians
// of its tile (no stage: a node's populations stay in its thread's registers),
// the tiles are many and independent, and the tile height follows the grid so
// that the SMs' shares are even. FP64 instructions per node are the strip
// kernel's within 2% (the tile's halo: densities on (32 + 4)(th + 4) points,
// phi and Laplacian on (32 + 2)(th + 2)). The node arithmetic is the same helper
// sequence in the same order, so the kernels give identical results.
//
// The FP32 step of a small grid (up to 4096 nodes per SM; both sides measured at the
// rule, plan_launch) is bound by latency: a row-pair CTA fills its pipeline for two
// to eight rows of its own, and pays twice the densities and potentials. A tile has
// no pipeline to fill. 512 x 128: 7.3 us a step by row pairs, 5.3 by tiles. Launched
// plainly: with programmatic launches, CTAs of the next step placed while this one
// runs share SMs that the rest then do without (512 x 128: 6.2 us; 1024 x 256:
// 11.6 against 10.0; FP64 at 128 x 128: 25 against 11).
//
// The FP32 fields (density, velocity, wall loads of the current state) take the
// same kernel: they read 36 B and write 12 B per node once, with no row
// pipeline to fill.
//
// Phases, a barrier after each: (1) densities and phi; (2) Laplacian; (3) force,
// collision, boundaries, push, diagnostics. CTAs stride over the tiles.
#pragma once

namespace lbm {

constexpr int T64_TX = 32, T64_MAX = 8;  // tile columns; most rows
constexpr int T64_AW = T64_TX + 4, T64_BW = T64_TX + 2;

template <typename real>
struct SmemT64 {
    real rho[T64_AW * (T64_MAX + 4)];
    real phi[T64_BW * (T64_MAX + 2)];
    real lap[T64_BW * (T64_MAX + 2)];
    real wv[T64_TX * T64_MAX];  // v_x of the rows next to the walls
    double red[T64_MAX][2];
    real ext[T64_MAX][4];
    int bad;
};

// Tile grid: th rows per tile, shifted one column left when the outlet column
// would open a tile (its stencil is its neighbour's), one row down when no height
// keeps the two rows next to a wall in one tile. CTAs stride over the tiles row of
// tiles by row of tiles. A tile with a pressure column costs more (its lanes
// extrapolate besides), and where the stride comes back to the same column of tiles
// within a few steps (456 CTAs over 3, 4, 6, 8, 12, 16 columns) the same CTAs would
// get such tiles again and again: in FP64 each row of tiles then starts rot tiles
// further on than the one before, as the host finds best (tile64_rotate; us per step
// without and with, 97 x 60000: 3283 and 2615; 250 x 24000: 2619 and 1832; 4096 x 512:
// 563 and 550). No one rotation fits all widths (2444 x 941: 986 with rot = 1, 620 with
// the one chosen). In FP32 it brings nothing, and its code costs 1 to 3% (512 x 128: 5.28
// and 5.45; 1024 x 256: 9.87 and 10.14).
struct T64Plan {
    int th, ntx, ntiles, sx, sy, rot;
};

// row pointers of a shared array as the 3 x 3 operands of the stencils
template <int SW, typename real>
__device__ __forceinline__ Row3<real> row3d(const real *a, int r, int c)
{
    const real *p = a + r * SW + c;
    return Row3<real>{p[-1], p[0], p[1]};
}

template <typename real, bool WALLS, bool PRES, int MODE, typename IX>
__global__ void __launch_bounds__(T64_TX *T64_MAX, 3) step_kernel_tile64(const KArgs<real> A, const T64Plan T)
{
    __shared__ SmemT64<real> S;
    const int tid = threadIdx.x, tx = tid & (T64_TX - 1), ty = tid >> 5, th = T.th, tn = T64_TX * th;
    const int nx = A.nx, ny = A.ny, P = A.pitch, rstride = 9 * P;
    const int yf0 = WALLS ? 1 : 0, yf1 = WALLS ? ny - 1 : ny;  // fluid rows yf0 .. yf1-1
    const real third = real(1.0 / 3.0);
    const Geom<real> G{A.fin, A.fout, nx, ny, A.W, P, A.rho_in_g, A.rho_in_l, A.rho_out_g, A.rho_out_l};
    Acc<real, 1> acc;
    acc.reset();

    // density and (want) phi of a stencil point (x, y) up to two nodes off the
    // lattice; a pressure column's density comes from its interior neighbour
    auto sum_at = [&](const real *p) {
        const real s = add_(add_(add_(p[0], p[P]), add_(p[2 * P], p[3 * P])),
                            add_(add_(p[4 * P], p[5 * P]), add_(p[6 * P], p[7 * P])));
        return add_(s, p[8 * P]);
    };
    auto column_of = [&](int x) {
        if (PRES) return min(max(x, 1), nx - 2);
        const int r = x < 0 ? x + nx : (x >= nx ? x - nx : x);
        return r >= 0 && r < nx ? r : ((x % nx) + nx) % nx;
    };
    const int cta = A.reverse ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;

    for (int t = cta; t < T.ntiles; t += gridDim.x) {
        const int by = t / T.ntx;
        int bx = t - by * T.ntx;
        if constexpr (PRES && MODE == MODE_STEP && sizeof(real) == 8) {
            if (T.rot) bx = (bx + by * T.rot) % T.ntx;
        }
        const int x0 = bx * T64_TX - T.sx, y0 = yf0 + by * th - T.sy;
        const int xa = x0 + tx, r = y0 + ty;
        const bool active = xa >= 0 && xa < nx && r >= yf0 && r < yf1;
        const bool pin = PRES && active && xa == 0, pout = PRES && active && xa == nx - 1;
        const bool anyp = pin || pout;

        // (1) densities, phi. Points beyond what the tile's nodes reach read a
        // clamped node's populations (finite, unused).
        auto density = [&](int c, int q) {  // local column -2 .. 33, row -2 .. th+1
            const int x = x0 + c, y = min(y0 + q, yf1 + 1);
            bool mir;
            const int row = map_row<WALLS>(y, ny, mir);
            real s = sum_at(G.fin + (IX)row * rstride + column_of(x));
            if (PRES && (x <= 0 || x >= nx - 1)) s = column_density(A, G, x >= nx - 1, s);
            return add_(s, mir ? A.wet : real(0));
        };
        real f[9];
        {
            const int row = min(max(r, yf0), yf1 - 1);
            const real *p = G.fin + (IX)row * rstride + column_of(xa);
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i] = __ldg(p + i * P);
        }
        for (int h = tid; h < T64_AW * (th + 4) - tn; h += tn) {
            int c, q;
            if (h < 4 * T64_AW) {
                const int k = h / T64_AW;
                c = h - k * T64_AW - 2;
                q = k < 2 ? k - 2 : th + k - 2;
            } else {
                const int k = (h - 4 * T64_AW) & 3;
                q = (h - 4 * T64_AW) >> 2;
                c = k < 2 ? k - 2 : T64_TX + k - 2;
            }
            const real v = density(c, q);
            S.rho[(q + 2) * T64_AW + c + 2] = v;
            if (c >= -1 && c <= T64_TX && q >= -1 && q <= th) S.phi[(q + 1) * T64_BW + c + 1] = eos_phi<real>(A, v);
        }
        {
            real s = add_(add_(add_(f[0], f[1]), add_(f[2], f[3])), add_(add_(f[4], f[5]), add_(f[6], f[7])));
            s = add_(s, f[8]);
            if (PRES && (xa <= 0 || xa >= nx - 1)) s = column_density(A, G, xa >= nx - 1, s);
            // a tile's rows beyond the fluid are its halo
            s = r < yf0 || r >= yf1 ? density(tx, ty) : add_(s, real(0));
            S.rho[(ty + 2) * T64_AW + tx + 2] = s;
            S.phi[(ty + 1) * T64_BW + tx + 1] = eos_phi<real>(A, s);
        }
        __syncthreads();

        // (2) Laplacian on the tile and one node around it
        auto lap = [&](int c, int q) {
            S.lap[(q + 1) * T64_BW + c + 1] = lap_stored<real>(row3d<T64_AW>(S.rho, q + 1, c + 2), row3d<T64_AW>(S.rho, q + 2, c + 2),
                                                         row3d<T64_AW>(S.rho, q + 3, c + 2));
        };
        lap(tx, ty);
        for (int h = tid; h < T64_BW * (th + 2) - tn; h += tn) {
            if (h < 2 * T64_BW) {
                const int k = h / T64_BW;
                lap(h - k * T64_BW - 1, k ? th : -1);
            } else {
                lap(((h - 2 * T64_BW) & 1) ? T64_TX : -1, (h - 2 * T64_BW) >> 1);
            }
        }
        __syncthreads();

        // (3) force, collision, push
        const int lc = pin ? tx + 1 : (pout ? tx - 1 : tx);  // a pressure column collides its neighbour
        const int ca = lc + 2, cb = lc + 1, qa = ty + 2, qb = ty + 1;
        real rho = real(0), vx = real(0);
        if (active) {
            rho = S.rho[qa * T64_AW + ca];
            real Fx, Fy;
            node_force(A, rho, row3d<T64_BW>(S.phi, qb - 1, cb), row3d<T64_BW>(S.phi, qb, cb),
                       row3d<T64_BW>(S.phi, qb + 1, cb), row3d<T64_BW>(S.lap, qb - 1, cb), row3d<T64_BW>(S.lap, qb, cb),
                       row3d<T64_BW>(S.lap, qb + 1, cb), Fx, Fy);
            const real jx = add_(add_(sub_(f[1], f[3]), sub_(f[5], f[6])), sub_(f[8], f[7]));
            const real jy = sub_(add_(sub_(f[2], f[4]), add_(f[5], f[6])), add_(f[7], f[8]));
            const real irho = rcp_(rho);
            const bool wall_row = WALLS && (r <= 2 || r >= ny - 3);
            real vy = real(0);
            if (MODE == MODE_FIELDS || anyp || wall_row) {
                const real ux = mul_(jx, irho), uy = mul_(jy, irho), hFi = mul_(irho, real(0.5));
                vx = fma_(hFi, Fx, ux);
                vy = fma_(hFi, Fy, uy);
            }
            const real rho_own = anyp ? S.rho[qa * T64_AW + tx + 2] : rho;
            if (MODE == MODE_STEP) {
                real fs[9];
                if (anyp) {
                    const real mvx = fma_(real(0.5), Fx, jx), mvy = fma_(real(0.5), Fy, jy);
                    column_extrapolate<real>(A, rho_own, rho, vx, vy, mvx, mvy, f, fs);
                } else {
                    const real mx = fma_(A.ushift, Fx, jx), my = fma_(A.ushift, Fy, jy);
                    if (A.mrt) {
                        real fe[9];
                        feq_pairs<real>(rho, mul_(mx, irho), mul_(my, irho), mx, my, fe);
                        mrt_relax<real, real>(A, f, fe, fs);
                    } else {
                        node_bgk(A, rho, irho, mx, my, f, fs);
                    }
                }
                real *const out = G.fout;
                const IX oi = (IX)r * rstride + xa;
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    int x = xa + ex_(i), y = r + ey_(i);
                    if (WALLS && (y == 0 || y == ny - 1)) {
                        out[oi + opp_(i) * P] = fs[i];  // half-way bounce-back
                        continue;
                    }
                    if (PRES) {
                        if (x < 0 || x >= nx) continue;  // leaves through the column
                    } else {
                        x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
                    }
                    if (!WALLS) y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
                    out[(IX)y * rstride + i * P + x] = fs[i];
                }
                // FP32: the mass as a compensated FP32 pair
                if constexpr (sizeof(real) == 4) two_sum_acc(acc.mhi, acc.mlo, rho_own);
                else acc.mass += rho_own;
                acc.range(rho);
            } else {
                // outputs may be absent; wall rows and the wall loads of a
                // pressure column are zero
                auto put = [&](real *o, int y, real v) {
                    if (o) o[(long long)y * nx + xa] = v;
                };
                put(A.o_rho, r, rho_own);
                put(A.o_vx, r, vx);
                put(A.o_vy, r, vy);
                if (WALLS && (r == 1 || r == ny - 2)) {
#pragma unroll
                    for (int side = 0; side < 2; ++side) {
                        if (r != (side ? ny - 2 : 1)) continue;
                        const int y = side ? ny - 1 : 0;
                        put(A.o_rho, y, real(0));
                        put(A.o_vx, y, real(0));
                        put(A.o_vy, y, real(0));
                        if (anyp) {
                            put(A.o_tw, side, real(0));
                            put(A.o_pw, side, real(0));
                        }
                    }
                }
            }
            if (WALLS && wall_row) S.wv[tid] = vx;
        }
        if (WALLS) {
            // wall shear: quadratic through v = 0 on the half-way plane and v at
            // distances 1/2 and 3/2 (both rows lie in this tile); wall pressure:
            // Eq. 2.4 in mesh units
            const bool low = y0 <= 1, high = y0 + th >= yf1;  // uniform
            if (low || high) {
                __syncthreads();
                if (active && !anyp) {
#pragma unroll
                    for (int side = 0; side < 2; ++side) {
                        if (r != (side ? ny - 2 : 1)) continue;
                        const real v2 = S.wv[tid + (side ? -T64_TX : T64_TX)];
                        const real tw = mul_(mul_(rho, A.nu), mul_(fma_(real(9), vx, -v2), third));
                        real grx, gry;
                        grad12<real>(row3d<T64_AW>(S.rho, qa - 1, ca), row3d<T64_AW>(S.rho, qa, ca),
                                     row3d<T64_AW>(S.rho, qa + 1, ca), grx, gry);
                        grx = mulk(grx, 1.0 / 12.0);
                        gry = mulk(gry, 1.0 / 12.0);
                        const real k2p0 = add_(S.phi[qb * T64_BW + cb], mulk(rho, 1.0 / 3.0));
                        const real tt = fma_(mul_(A.kappa, rho), -lap_of_stored<real>(S.lap[qb * T64_BW + cb]), k2p0);
                        const real pw = fma_(fma_(grx, grx, mul_(gry, gry)), mul_(real(-0.5), A.kappa), tt);
                        if (MODE == MODE_STEP) {
                            acc.J += (double)tw;
                            acc.tmin = fmin(acc.tmin, tw); acc.tmax = fmax(acc.tmax, tw);
                            acc.pmin = fmin(acc.pmin, pw); acc.pmax = fmax(acc.pmax, pw);
                        } else {
                            if (A.o_tw) A.o_tw[side * nx + xa] = tw;
                            if (A.o_pw) A.o_pw[side * nx + xa] = pw;
                        }
                    }
                }
            }
        }
        __syncthreads();  // the shared arrays serve the next tile
    }
    if constexpr (MODE == MODE_STEP) {

    // fixed-order reduction: lanes by butterflies, then the warps in order
    const int lane = tid & 31, warp = tid >> 5;
    real e[4] = {acc.tmin, acc.tmax, acc.pmin, acc.pmax};
    const bool anyw = __any_sync(0xffffffffu, e[0] < real(INFINITY) || e[1] > -real(INFINITY) ||
                                                  e[2] < real(INFINITY) || e[3] > -real(INFINITY) || acc.J != 0.0);
    const bool wbad = __any_sync(0xffffffffu, acc.bad());
    if constexpr (sizeof(real) == 4) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float h2 = __shfl_xor_sync(0xffffffffu, acc.mhi, o), l2 = __shfl_xor_sync(0xffffffffu, acc.mlo, o);
            two_sum_acc(acc.mhi, acc.mlo, h2);
            acc.mlo = __fadd_rn(acc.mlo, l2);
        }
        acc.mass = (double)acc.mhi + (double)acc.mlo;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if constexpr (sizeof(real) == 8) acc.mass += __shfl_xor_sync(0xffffffffu, acc.mass, o);
        if (anyw) {
            acc.J += __shfl_xor_sync(0xffffffffu, acc.J, o);
            e[0] = fmin(e[0], __shfl_xor_sync(0xffffffffu, e[0], o));
            e[1] = fmax(e[1], __shfl_xor_sync(0xffffffffu, e[1], o));
            e[2] = fmin(e[2], __shfl_xor_sync(0xffffffffu, e[2], o));
            e[3] = fmax(e[3], __shfl_xor_sync(0xffffffffu, e[3], o));
        }
    }
    if (tid == 0) S.bad = 0;
    __syncthreads();
    if (lane == 0) {
        S.red[warp][0] = acc.mass;
        S.red[warp][1] = acc.J;
        for (int k = 0; k < 4; ++k) S.ext[warp][k] = e[k];
        if (wbad) atomicOr(&S.bad, 1);
    }
    __syncthreads();
    if (tid == 0) {
        double m = 0.0, j = 0.0;
        for (int w = 0; w < th; ++w) {
            m += S.red[w][0];
            j += S.red[w][1];
            e[0] = fmin(e[0], S.ext[w][0]); e[1] = fmax(e[1], S.ext[w][1]);
            e[2] = fmin(e[2], S.ext[w][2]); e[3] = fmax(e[3], S.ext[w][3]);
        }
        A.mass_part[cta] = m;
        A.J_acc[cta] += j;
        real *ex = A.ext + 4 * cta;
        ex[0] = fmin(ex[0], e[0]); ex[1] = fmax(ex[1], e[1]);
        ex[2] = fmin(ex[2], e[2]); ex[3] = fmax(ex[3], e[3]);
        if (S.bad) atomicOr(A.err, 1);
    }
    }
}

}  // namespace lbm
