"""Heights whose bands of one CTA's share of rows would leave a last band of a few
rows: the FP32 row pairs with the bands of the default plan against one row per
thread over another CTA count (other bands and cuts), bit for bit.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,walls,bc_x", [(1999, 1500, True, False), (1999, 1500, True, True), (1180, 741, False, False),
                                              (2053, 398, False, False), (5343, 1244, False, True), (20000, 40, True, True)])
def test_bands_do_not_show(orc, nx, ny, walls, bc_x):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    import paper_2103_08301_gb300 as lbm
    kw = dict(walls=walls, bc_x=bc_x, T_over_Tc=0.85, kappa=0.5, dp=1e-3 if bc_x else 0.0, gx=1e-6)
    g, l, _ = orc.Setup(nx=nx, ny=ny, **kw).coexistence()
    rho0 = synth.disk_rho0(nx, ny, min(nx, ny) / 4, l, g, noise=1e-3, seed=nx)
    out = []
    for opts in ({}, {"LBM_OPT_ROWS2": 0, "LBM_OPT_CTAS_PER_SM": 3}):
        with lbm.Lattice(nx, ny, rho0, precision=32, **kw) as lat:
            for k, v in opts.items():
                lat.set_option(getattr(lbm, k), v)
            lat.step(9)
            out.append((lat.populations(), lat.diag()))
    y, x = slice(1, ny - 1) if walls else slice(None), slice(1, nx - 1) if bc_x else slice(None)
    assert np.array_equal(out[0][0][:, y, x].view(np.uint32), out[1][0][:, y, x].view(np.uint32))
    for k in ("tau_wall_min", "tau_wall_max", "p_wall_min", "p_wall_max", "nan_detected", "step"):
        assert out[0][1][k] == out[1][1][k], k
    # up to 16 rows of a lane are added in FP32 first: 16 x 2^-24
    assert abs(out[0][1]["mass"] / out[1][1]["mass"] - 1) <= 1e-6
