"""The FP32 row-pair step where its loads change: periodic widths that are not
a multiple of 4 (rows start at any 4-byte offset and the strips at the seam
wrap), strips whose last lane is the only one, and general-geometry (mask)
steps of the same sizes, bit for bit against the kernels of one row per thread.
The node arithmetic is the same in the same order, so no tolerance is needed.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

# nx, ny, walls
WIDTHS = [(1, 7, False), (2, 2, False), (3, 9, True), (5, 1, False), (121, 14, False), (123, 9, True),
          (125, 33, False), (127, 6, True), (249, 21, False), (997, 40, True), (1999, 77, False)]


def _run(lbm, nx, ny, rho0, opts, **kw):
    with lbm.Lattice(nx, ny, rho0, precision=32, T_over_Tc=0.85, kappa=0.5, **kw) as lat:
        for k, v in opts.items():
            lat.set_option(getattr(lbm, k), v)
        lat.step(37)
        return lat.populations(), lat.diag()


CASES = [w + (False,) for w in WIDTHS] + [w + (True,) for w in WIDTHS if w[0] > 100]


@pytest.mark.parametrize("nx,ny,walls,mask", CASES)
def test_row_pairs_on_odd_periodic_widths(orc, nx, ny, walls, mask):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    import paper_2103_08301_gb300 as lbm
    g, l, _ = orc.Setup(nx=nx, ny=ny, walls=walls, T_over_Tc=0.85, kappa=0.5).coexistence()
    rho0 = synth.disk_rho0(nx, ny, max(nx, ny) / 4, l, g, noise=1e-3, seed=nx)
    kw = dict(walls=walls, gx=1e-6)
    solid = np.zeros((ny, nx), np.uint8)
    if mask:
        # solid nodes in the flow: at both ends of a row, a single one, a pair
        solid[ny // 2, [0, nx // 2, nx - 1]] = 1
        solid[ny // 3, nx // 3:nx // 3 + 2] = 1
        kw["mask"] = solid
    pairs, d1 = _run(lbm, nx, ny, rho0, {}, **kw)
    rows, d0 = _run(lbm, nx, ny, rho0, {"LBM_OPT_ROWS2": 0}, **kw)
    fluid = solid == 0
    if walls:
        fluid[0] = fluid[-1] = False
    assert np.array_equal(pairs[:, fluid].view(np.uint32), rows[:, fluid].view(np.uint32))
    assert d1["nan_detected"] == d0["nan_detected"]
    # row pairs add up to 16 rows of a lane in FP32 before their
    # compensated sum: relative error up to 16 x 2^-24
    assert abs(d1["mass"] / d0["mass"] - 1) <= 1e-6
