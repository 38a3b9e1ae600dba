"""Solid nodes in FP32 on either side of the rule that picks row pairs or the
general-geometry kernels (a node per thread): populations and extrema bit for bit
against the latter. The route is read from a checkpoint's header (CTAs whose partials
it holds): row pairs run 5 CTAs an SM at most.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


# nx, ny, walls, pressure columns, row pairs
@pytest.mark.parametrize("nx,ny,walls,bc_x,pairs", [
    (256, 256, False, False, False), (1024, 1024, False, False, True), (127, 5000, False, False, False),
    (97, 6000, True, True, False), (97, 1000, True, True, True), (97, 60000, True, False, True),
    (250, 3000, False, True, False), (1024, 256, True, True, True), (130, 4000, True, False, False),
    (1999, 501, False, False, True), (1021, 1101, False, False, True), (1337, 777, True, False, True)])
def test_route_and_bits(orc, nx, ny, walls, bc_x, pairs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    import paper_2103_08301_gb300 as lbm
    kw = dict(walls=walls, bc_x=bc_x, T_over_Tc=0.85, kappa=0.5, dp=1e-3 if bc_x else 0.0, gx=1e-6)
    g, l, _ = orc.Setup(nx=nx, ny=ny, **kw).coexistence()
    rho0 = synth.disk_rho0(nx, ny, min(nx, ny) / 4, l, g, noise=1e-3, seed=nx)
    mask = np.zeros((ny, nx), np.uint8)
    mask[ny // 2:ny // 2 + 3, nx // 2:nx // 2 + 5] = mask[ny // 3, nx // 3] = 1
    if not bc_x:  # the ends of rows, where odd widths wrap
        mask[ny // 2 + 9, [0, nx - 1]] = mask[ny - 3, nx - 2:] = 1
    out = []
    for opts in ({}, {"LBM_OPT_ROWS2": 0}):
        with lbm.Lattice(nx, ny, rho0, precision=32, mask=mask, **kw) as lat:
            for k, v in opts.items():
                lat.set_option(getattr(lbm, k), v)
            lat.step(9)
            ctas, general = int(lat.checkpoint()[8:32].view(np.int32)[5]), lat.launch_info()["ctas"]
            assert (ctas != general) == (pairs and not opts), (ctas, general)
            out.append((lat.populations(), lat.diag()))
    fluid = mask == 0
    if walls:
        fluid[0] = fluid[-1] = False
    if bc_x:
        fluid[:, 0] = fluid[:, -1] = False
    assert np.array_equal(out[0][0][:, fluid].view(np.uint32), out[1][0][:, fluid].view(np.uint32))
    for k in ("tau_wall_min", "tau_wall_max", "p_wall_min", "p_wall_max", "nan_detected", "step"):
        assert out[0][1][k] == out[1][1][k], k
    # up to 16 rows of a lane are added in FP32 first: 16 x 2^-24
    assert abs(out[0][1]["mass"] / out[1][1]["mass"] - 1) <= 1e-6
