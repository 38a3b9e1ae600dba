"""Odd periodic widths in FP32: one row per thread where its wider strips are fewer
than the row pairs' (told by the work units, strips times rows), row pairs
elsewhere; populations bit for bit against row pairs (an explicit strip width).
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


# nx, ny, walls, strips
@pytest.mark.parametrize("nx,ny,walls,strips", [
    (125, 6400, False, 1), (127, 6300, True, 1), (121, 6500, True, 1), (250, 3200, False, 3), (250, 3200, True, 3),
    (253, 24000, False, 2), (253, 8000, True, 2), (253, 8000, False, 3), (381, 15748, True, 4), (1999, 400, True, 17)])
def test_route_and_bits(orc, nx, ny, walls, strips):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    import paper_2103_08301_gb300 as lbm
    kw = dict(walls=walls, T_over_Tc=0.85, kappa=0.5, gx=1e-6)
    g, l, _ = orc.Setup(nx=nx, ny=ny, **kw).coexistence()
    rho0 = synth.disk_rho0(nx, ny, min(nx, ny) / 4, l, g, noise=1e-3, seed=nx)
    out = []
    for strip in (0, 124):
        with lbm.Lattice(nx, ny, rho0, precision=32, **kw) as lat:
            if strip:
                lat.set_option(lbm.LBM_OPT_STRIP, strip)
            rows = ny - 2 * walls
            assert lat.launch_info()["units"] == rows * (-(-nx // 124) if strip else strips)
            lat.step(9)
            out.append((lat.populations(), lat.diag()))
    y = slice(1, ny - 1) if walls else slice(None)
    assert np.array_equal(out[0][0][:, y].view(np.uint32), out[1][0][:, y].view(np.uint32))
    for k in ("tau_wall_min", "tau_wall_max", "p_wall_min", "p_wall_max", "nan_detected", "step"):
        assert out[0][1][k] == out[1][1][k], k
    # up to 16 rows of a lane are added in FP32 first: 16 x 2^-24
    assert abs(out[0][1]["mass"] / out[1][1]["mass"] - 1) <= 1e-6
