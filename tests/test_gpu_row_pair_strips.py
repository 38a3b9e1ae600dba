"""The FP32 row-pair step on small grids, which take the tile kernel unless a strip
width is given: an explicit one keeps these on row pairs, and the launch geometry
says so. Odd periodic widths (rows start at any 4-byte offset, the strips at the
seam wrap) and tiny channels against the kernel of one row per thread; prefetch and
programmatic launches against none. The node arithmetic is the same in the same
order, so no tolerance is needed for populations.
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


def _run(lbm, nx, ny, rho0, steps, opts, **kw):
    with lbm.Lattice(nx, ny, rho0, precision=32, T_over_Tc=0.85, kappa=0.5, **kw) as lat:
        lat.set_option(lbm.LBM_OPT_STRIP, 124)
        for k, v in opts.items():
            lat.set_option(getattr(lbm, k), v)
        info = lat.launch_info()
        rows = ny - 2 if kw.get("walls") else ny
        assert info["threads"] == 128 and info["staged"] and info["units"] % rows == 0
        assert info["units"] // rows in (-(-nx // 124), -(-nx // 120))  # strips (narrower: the outlet's rule), not tiles
        lat.step(steps)
        return lat.populations(), lat.diag()


def _bits(a, b):
    return np.array_equal(a.view(np.uint32), b.view(np.uint32))


# nx, ny, walls, pressure columns
SIZES = [(1, 7, False, False), (2, 2, False, False), (3, 9, True, False), (5, 1, False, False), (121, 14, False, False),
         (123, 9, True, False), (125, 33, False, False), (127, 6, True, False), (249, 21, False, False),
         (997, 40, True, False), (1999, 77, False, False), (4, 4, True, True), (5, 7, True, True), (130, 5, True, True),
         (125, 12, True, True), (12, 5, False, False)]


@pytest.mark.parametrize("nx,ny,walls,bc_x", SIZES)
def test_row_pairs_match_one_row_per_thread(orc, lbm, nx, ny, walls, bc_x):
    g, l, _ = orc.Setup(nx=nx, ny=ny, walls=walls, bc_x=bc_x, T_over_Tc=0.85, kappa=0.5).coexistence()
    rho0 = synth.disk_rho0(nx, ny, max(nx, ny) / 4, l, g, noise=1e-3, seed=nx)
    kw = dict(walls=walls, bc_x=bc_x, gx=1e-6)
    pairs, d1 = _run(lbm, nx, ny, rho0, 37, {}, **kw)
    rows, d0 = _run(lbm, nx, ny, rho0, 37, {"LBM_OPT_ROWS2": 0}, **kw)
    fluid = np.ones((ny, nx), bool)
    if walls:
        fluid[0] = fluid[-1] = False
    if bc_x:
        fluid[:, 0] = fluid[:, -1] = False
    assert _bits(pairs[:, fluid], rows[:, fluid])
    assert d1["nan_detected"] == d0["nan_detected"]
    # up to 16 rows of a lane are added in FP32 before their compensated sum: 16 x 2^-24
    assert abs(d1["mass"] / d0["mass"] - 1) <= 1e-6


@pytest.mark.parametrize("opts", [{"LBM_OPT_PREFETCH": 1}, {"LBM_OPT_PREFETCH": 3}, {"LBM_OPT_PDL": 0}, {"LBM_OPT_TMA": 0}])
@pytest.mark.parametrize("walls,graphs", [(True, 0), (True, 64), (False, 0)])
def test_launch_options_change_nothing(orc, lbm, opts, walls, graphs):
    import torch
    nx, ny = 1024, 128
    g, l, _ = orc.Setup(nx=nx, ny=ny, walls=walls, bc_x=walls, T_over_Tc=0.85, kappa=0.5).coexistence()
    rho0 = synth.airway_rho0(nx, ny, 6, 256, 96, l, g, noise=1e-3, seed=2) if walls else \
        synth.disk_rho0(nx, ny, 40, l, g, noise=1e-3, seed=2)
    kw = dict(walls=walls, bc_x=walls, dp=1e-3 if walls else 0.0)
    out = []
    for o in (opts, {}):
        out.append(_run(lbm, nx, ny, rho0, 301, dict(o, LBM_OPT_GRAPH_STEPS=graphs), stream=torch.cuda.Stream(), **kw))
    assert _bits(out[0][0], out[1][0])
    assert out[0][1] == out[1][1]
