"""Restoring a checkpoint takes the partials that its header counts: what lies beyond
them in the file (an older plan's remains) is no part of the totals.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

MAX_CTAS = 8192  # partial slots of a file: mass and wall shear (8 bytes each), four extrema


@pytest.mark.parametrize("precision", [32, 64])
def test_slots_beyond_the_count_are_not_added(orc, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    import paper_2103_08301_gb300 as lbm
    nx, ny = 512, 128
    kw = dict(walls=True, bc_x=True, T_over_Tc=0.85, kappa=0.5, dp=1e-3)
    g, l, _ = orc.Setup(nx=nx, ny=ny, **kw).coexistence()
    rho0 = synth.airway_rho0(nx, ny, 6, 128, 48, l, g)
    with lbm.Lattice(nx, ny, rho0, precision=precision, **kw) as lat:
        lat.step(20)
        want = lat.diag()
        ck = lat.checkpoint()
        ctas = int(ck[8:32].view(np.int32)[5])
        sz = precision // 8
        parts = len(ck) - 4 - MAX_CTAS * (16 + 4 * sz)  # before them: header and populations
        shear = ck[parts + MAX_CTAS * 8:parts + MAX_CTAS * 16].copy().view(np.float64)
        assert abs(shear[:ctas].sum() - want["wall_shear_sum"]) <= 1e-12 * np.abs(shear[:ctas]).sum()
        shear[ctas:] = 1.0
        ck[parts + MAX_CTAS * 8:parts + MAX_CTAS * 16] = shear.view(np.uint8)
        lat.restore(ck)
        assert lat.diag() == want
