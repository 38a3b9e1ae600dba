"""The FP64 tile kernel at the edges of its tiles (32 columns, 2 to 8 rows):
the outlet column opening a tile (nx = 33, 65), remainders of one row and
column, heights where no tile height keeps the wall rows together (843), grids
smaller than a tile and its halo, and 64-bit-free strides over several tiles
per CTA, against the FP64 oracle.

Twenty steps of about 130 operations per node round at 1.1e-16 each, on values
up to the largest population: 1e-12 of it leaves two orders of room. The wall
loads divide by the vapour's density (0.03) and difference neighbouring rows:
1e-9 of their largest value.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

# nx, ny, walls, columns, tau, wetting
GRIDS = [(33, 18, True, True, 1.0, 0.0), (65, 11, True, True, 1.1, 0.002), (32, 9, True, False, 1.0, 0.001),
         (40, 843, True, True, 1.0, 0.0), (5, 4, True, True, 1.0, 0.0), (4, 5, True, False, 1.2, 0.0),
         (1, 7, False, False, 1.0, 0.0), (33, 1, False, False, 1.0, 0.0), (31, 10, False, True, 1.0, 0.0),
         (129, 67, False, False, 1.3, 0.0), (700, 300, True, True, 1.0, 0.0)]


@pytest.mark.parametrize("nx,ny,walls,bc_x,tau,wet", GRIDS)
def test_tiles_match_the_oracle(orc, nx, ny, walls, bc_x, tau, wet):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    import paper_2103_08301_gb300 as lbm
    kw = dict(walls=walls, bc_x=bc_x, T_over_Tc=0.85, kappa=0.5, tau=tau, dp=2e-4 if bc_x else 0.0, gx=1e-6)
    s = orc.Setup(nx=nx, ny=ny, wet=wet, **kw)
    g, l, _ = s.coexistence()
    if walls:
        rho0 = synth.airway_rho0(nx, ny, max(1, ny // 16), nx // 4, max(1, nx // 6), l, g, noise=1e-3, seed=2)
    else:
        rho0 = synth.disk_rho0(nx, ny, max(nx, ny) / 4, l, g, noise=1e-3, seed=2)
    f, d_ref = orc.run(s, orc.init(s, rho0), 20)
    with lbm.Lattice(nx, ny, rho0, precision=64, wetting=wet, **kw) as lat:
        lat.step(20)
        got, fld, d = lat.populations(), lat.fields(), lat.diag()
    fluid = np.ones((ny, nx), bool)
    if walls:
        fluid[0] = fluid[-1] = False
    if bc_x:
        fluid[:, 0] = fluid[:, -1] = False
    scale = np.abs(f[:, fluid]).max()
    assert np.abs(got - f)[:, fluid].max() <= 1e-12 * scale
    ref = orc.fields(s, f)
    assert np.abs(fld["rho"] - ref["rho"]).max() <= 1e-12 * np.abs(ref["rho"]).max()
    for k in ("vx", "vy"):
        assert np.abs(fld[k] - ref[k]).max() <= 1e-11
    if walls:
        for k in ("tau_wall", "p_wall"):
            assert np.abs(fld[k] - ref[k]).max() <= 1e-9 * np.abs(ref[k]).max() + 1e-15
    assert abs(d["mass"] / d_ref["mass"] - 1) <= 1e-12
