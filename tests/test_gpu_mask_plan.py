"""The plan of the FP32 step with solid nodes: strips over as many CTAs as stay
resident, whatever the options that concern other kernels say. The CTA count is read
from a checkpoint's header (the partials' count), the populations bit for bit.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_tile_option_leaves_the_masked_plan_alone(orc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    import paper_2103_08301_gb300 as lbm
    nx, ny = 1024, 256
    kw = dict(walls=True, bc_x=True, T_over_Tc=0.85, kappa=0.5, dp=1e-3)
    g, l, _ = orc.Setup(nx=nx, ny=ny, **kw).coexistence()
    rho0 = synth.airway_rho0(nx, ny, 12, 256, 64, l, g, noise=1e-3, seed=1)
    mask = np.zeros((ny, nx), np.uint8)
    mask[1:40, 500:540] = mask[ny - 30:ny - 1, 500:540] = 1
    out = []
    for tile in (0, 1):
        with lbm.Lattice(nx, ny, rho0, precision=32, mask=mask, **kw) as lat:
            lat.set_option(lbm.LBM_OPT_TILE, tile)
            lat.step(37)
            ctas = int(lat.checkpoint()[8:32].view(np.int32)[5])
            out.append((ctas, lat.populations(), lat.diag()))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert out[0][0] == out[1][0] == 5 * sms  # 5 CTAs of 128 threads (launch bounds) fit an SM
    assert np.array_equal(out[0][1].view(np.uint32), out[1][1].view(np.uint32))
    assert out[0][2] == out[1][2]
