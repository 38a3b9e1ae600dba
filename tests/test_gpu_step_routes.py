"""FP32 steps by the kernel that a size selects, bit for bit against the one it
replaces (the same node arithmetic in the same order, so populations, fields and
extrema need no tolerance; the sums are taken in another order).

Small grids: tiles of one node per thread against row pairs (an explicit strip
width selects those), at the edges of tiles and strips. Long in-place channels:
row pairs in place against the two-array step, with and without walls, over
strips and segments that the grid does not divide.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    import paper_2103_08301_gb300 as m
    return m


def _bits(a, b):
    return np.array_equal(np.ascontiguousarray(a).view(np.uint32), np.ascontiguousarray(b).view(np.uint32))


def _same(lbm, a, b, fluid, steps, mass_tol=1e-6):
    """mass_tol: up to 16 rows of a lane are added in FP32 first, 16 x 2^-24."""
    (fa, Fa, da), (fb, Fb, db) = a, b
    assert _bits(fa[:, fluid], fb[:, fluid])
    for k in ("rho", "vx", "vy", "tau_wall", "p_wall"):
        assert _bits(Fa[k], Fb[k]), k
    for k in ("tau_wall_min", "tau_wall_max", "p_wall_min", "p_wall_max", "nan_detected", "step"):
        assert da[k] == db[k], k
    assert abs(da["mass"] / db["mass"] - 1) <= mass_tol
    nw = 2 * fluid.shape[1] * steps * max(abs(da["tau_wall_min"]), abs(da["tau_wall_max"])) if da["tau_wall_max"] >= \
        da["tau_wall_min"] else 0.0
    # FP64 sums of 2 nx steps FP32 terms
    assert abs(da["wall_shear_sum"] - db["wall_shear_sum"]) <= 1e-10 * nw + 1e-15


def _rho0(orc, nx, ny, walls, bc):
    g, l, _ = orc.Setup(nx=nx, ny=ny, walls=walls, bc_x=bc, T_over_Tc=0.85, kappa=0.5).coexistence()
    if walls:
        return synth.airway_rho0(nx, ny, max(1, ny // 16), nx // 4, max(1, nx // 6), l, g, noise=1e-3, seed=nx)
    return synth.disk_rho0(nx, ny, max(nx, ny) / 4, l, g, noise=1e-3, seed=nx)


def _fluid(nx, ny, walls, bc):
    m = np.ones((ny, nx), bool)
    if walls:
        m[0] = m[-1] = False
    if bc:
        m[:, 0] = m[:, -1] = False
    return m


# nx, ny, walls, columns, tau, wetting, MRT
SMALL = [(33, 18, True, True, 1.0, 0.0, False), (65, 11, True, True, 1.1, 0.002, True), (5, 4, True, True, 1.0, 0.0, False),
         (4, 5, True, False, 1.2, 0.0, False), (7, 1, False, False, 1.0, 0.0, False), (2, 2, False, False, 1.0, 0.0, False),
         (40, 843, True, True, 1.0, 0.0, False), (31, 10, False, True, 1.0, 0.0, False),
         (129, 67, False, False, 1.3, 0.0, True), (997, 300, True, True, 1.0, 0.0, False),
         (2048, 304, True, True, 1.0, 0.0, False), (2048, 305, True, True, 1.0, 0.0, False)]


@pytest.mark.parametrize("nx,ny,walls,bc_x,tau,wet,mrt", SMALL)
def test_small_grids_step_by_tiles(orc, lbm, nx, ny, walls, bc_x, tau, wet, mrt):
    rho0 = _rho0(orc, nx, ny, walls, bc_x)
    kw = dict(walls=walls, bc_x=bc_x, T_over_Tc=0.85, kappa=0.5, tau=tau, dp=2e-4 if bc_x else 0.0, gx=1e-6)
    if mrt:
        kw.update(collision="mrt", s_e=1.2, s_eps=1.54, s_j=1 / tau, s_q=1.1)
    steps = 41
    out = []
    for strip in (0, 124):
        with lbm.Lattice(nx, ny, rho0, precision=32, wetting=wet, **kw) as lat:
            if strip:
                lat.set_option(lbm.LBM_OPT_STRIP, strip)
            lat.step(steps)
            out.append((lat.populations(), lat.fields(), lat.diag()))
    _same(lbm, out[0], out[1], _fluid(nx, ny, walls, bc_x), steps)


@pytest.mark.parametrize("walls", [True, False])
def test_row_pairs_tensor_loads_match_plane_copies(orc, lbm, walls):
    """The row-pair step's two stagings, on a grid that tiles would take."""
    nx, ny = 512, 64
    rho0 = _rho0(orc, nx, ny, walls, walls)
    kw = dict(walls=walls, bc_x=walls, T_over_Tc=0.85, kappa=0.5, dp=1e-3 if walls else 0.0)
    out = []
    for tma in (1, 0):
        with lbm.Lattice(nx, ny, rho0, precision=32, **kw) as lat:
            lat.set_option(lbm.LBM_OPT_STRIP, 124)
            lat.set_option(lbm.LBM_OPT_TMA, tma)
            lat.step(40)
            out.append((lat.populations(), lat.fields(), lat.diag()))
    _same(lbm, out[0], out[1], _fluid(nx, ny, walls, walls), 40)


@pytest.mark.parametrize("nx,ny,walls", [(4096, 1100, True), (3997, 1203, False), (1324, 4001, True)])
def test_long_channels_step_in_place_by_row_pairs(orc, lbm, nx, ny, walls):
    rho0 = _rho0(orc, nx, ny, walls, True)
    kw = dict(walls=walls, bc_x=True, T_over_Tc=0.85, kappa=0.5, dp=1e-3)
    out = []
    for inplace in (True, False):
        with lbm.Lattice(nx, ny, rho0, precision=32, inplace=inplace, **kw) as lat:
            if inplace:
                assert lat.launch_info()["staged"]  # row pairs, not tiles
            lat.step(9)  # ends in the odd-parity layout
            out.append((lat.populations(), lat.fields(), lat.diag()))
    _same(lbm, out[0], out[1], _fluid(nx, ny, walls, True), 9)
