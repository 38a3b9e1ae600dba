"""More tiles than CTAs between pressure columns, where each row of tiles starts one
tile further on: every node is stepped once. FP64 by tiles against strips (an
explicit strip width), bit for bit: the same node arithmetic in the same order.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,walls", [(20, 5000, True), (64, 3000, False), (97, 3003, True), (125, 2402, True),
                                         (250, 1204, True), (257, 1204, False), (1500, 242, True)])
def test_rotated_tile_rows_step_every_node(orc, nx, ny, walls):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    import paper_2103_08301_gb300 as lbm
    kw = dict(walls=walls, bc_x=True, T_over_Tc=0.85, kappa=0.5, dp=1e-4)
    g, l, _ = orc.Setup(nx=nx, ny=ny, **kw).coexistence()
    rho0 = synth.disk_rho0(nx, ny, min(nx, ny) / 4, l, g, noise=1e-3, seed=nx)
    out = []
    for strip in (0, 128):
        with lbm.Lattice(nx, ny, rho0, precision=64, **kw) as lat:
            if strip:
                lat.set_option(lbm.LBM_OPT_STRIP, strip)
            else:
                lat.set_option(lbm.LBM_OPT_CTAS_PER_SM, 1)  # fewer CTAs than tiles, by tiles
                info = lat.launch_info()
                assert info["units"] > info["ctas"] and info["units"] % -(-(nx + (nx % 32 == 1)) // 32) == 0
            lat.step(9)
            out.append((lat.populations(), lat.fields(), lat.diag()))
    (fa, Fa, da), (fb, Fb, db) = out
    y = slice(1, ny - 1) if walls else slice(None)
    assert np.array_equal(fa[:, y, 1:-1].view(np.uint64), fb[:, y, 1:-1].view(np.uint64))
    for k in ("rho", "vx", "vy", "tau_wall", "p_wall"):
        assert np.array_equal(Fa[k].view(np.uint64), Fb[k].view(np.uint64)), k
    for k in ("tau_wall_min", "tau_wall_max", "p_wall_min", "p_wall_max", "nan_detected", "step"):
        assert da[k] == db[k], k
    # sums of FP64 terms in another order
    assert abs(da["mass"] / db["mass"] - 1) <= 1e-12
