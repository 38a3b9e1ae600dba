"""In-place FP32 channels long enough to step by row pairs, bit for bit against
two-array contexts (the same node arithmetic in the same order; the sums are
taken in another order).

Widths that leave a last strip of two columns: the outlet column's density comes
from column nx-2, which then is another CTA's. Every part of the step that small
grids, which take the tiles, cannot reach: a wetting offset, MRT, Peng-Robinson,
graph replay and a checkpoint taken in the odd-parity layout.
"""
import ctypes as C

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


CS = dict(T_over_Tc=0.85, kappa=0.5, dp=1e-3)
PR = dict(eos="pr", a=2 / 49, b=2 / 21, T_over_Tc=0.8, k=1.0, kappa=0.01, tau=1.2, dp=1e-4)
MRT = dict(tau=1.2, collision="mrt", s_e=1 / 1.2, s_eps=1.54, s_q=1 / 1.2, s_j=1 / 1.2)


def _rho0(orc, nx, ny, walls, phys):
    kw = {k: v for k, v in phys.items() if k not in ("wetting", "collision") and not k.startswith("s_")}
    g, l, _ = orc.Setup(nx=nx, ny=ny, walls=walls, bc_x=True, **kw).coexistence()
    if walls:
        # a plug in the channel and one that reaches the outlet, films along the walls
        a = synth.airway_rho0(nx, ny, ny // 16, nx // 4, nx // 6, l, g, noise=1e-3, seed=nx)
        return np.maximum(a, synth.airway_rho0(nx, ny, ny // 16, nx - 40, 30, l, g, noise=1e-3, seed=ny))
    return np.maximum(synth.disk_rho0(nx, ny, ny / 4, l, g, noise=1e-3, seed=nx),
                      synth.disk_rho0(nx, ny, ny / 5, l, g, noise=1e-3, seed=ny, centre=(nx - 30.0, ny / 3)))


def _state(lbm, lat, walls):
    """Populations of the nodes between the boundaries as integers on the device, and the report."""
    import torch
    f = torch.empty((9, lat.ny, lat.nx), dtype=torch.float32, device="cuda")
    assert lbm.lib().lbm_populations(lat.ctx, C.c_void_p(f.data_ptr())) == lbm.LBM_OK
    y = slice(1, lat.ny - 1) if walls else slice(None)
    return f[:, y, 1:lat.nx - 1].contiguous().view(torch.int32), lat.diag()


def _same(a, b):
    import torch
    (fa, da), (fb, db) = a, b
    assert torch.equal(fa, fb), f"{int((fa != fb).sum())} populations differ"
    for k in ("tau_wall_min", "tau_wall_max", "p_wall_min", "p_wall_max", "nan_detected", "step"):
        assert da[k] == db[k], k
    assert not da["nan_detected"]


def _in_place(lbm, nx, ny, rho0, **kw):
    lat = lbm.Lattice(nx, ny, rho0, precision=32, bc_x=True, inplace=True, **kw)
    info = lat.launch_info()
    assert info["staged"] and info["units"] == -(-nx // 120) * (ny - 2 if kw["walls"] else ny)  # row pairs, not tiles
    return lat


# 4082 = 34 * 120 + 2 and 8162 = 68 * 120 + 2
@pytest.mark.parametrize("nx,ny,walls,phys", [
    (4082, 1100, True, CS), (4082, 1100, False, CS), (8162, 600, True, CS),
    (4082, 1100, True, dict(CS, wetting=0.003)), (4082, 1100, True, dict(CS, **MRT)), (4082, 1100, False, dict(CS, **MRT)),
    (4082, 1100, True, PR)])
def test_two_column_last_strip(orc, lbm, nx, ny, walls, phys):
    rho0 = _rho0(orc, nx, ny, walls, phys)
    with lbm.Lattice(nx, ny, rho0, precision=32, walls=walls, bc_x=True, **phys) as lat:
        lat.step(301)  # an odd number: the in-place array ends in the odd-parity layout
        ref = _state(lbm, lat, walls)
    for _ in range(2):
        with _in_place(lbm, nx, ny, rho0, walls=walls, **phys) as lat:
            lat.step(301)
            _same(_state(lbm, lat, walls), ref)


def test_graph_replay_and_odd_parity_checkpoint(orc, lbm):
    import torch
    nx, ny = 4082, 1100
    rho0 = _rho0(orc, nx, ny, True, CS)
    with lbm.Lattice(nx, ny, rho0, precision=32, walls=True, bc_x=True, **CS) as lat:
        lat.step(195)
        ref = _state(lbm, lat, True)
    with _in_place(lbm, nx, ny, rho0, walls=True, stream=torch.cuda.Stream(), **CS) as lat:
        lat.set_option(lbm.LBM_OPT_GRAPH_STEPS, 64)
        lat.step(1)    # the next run starts in the odd-parity layout
        lat.step(130)
        lat.step(64)
        _same(_state(lbm, lat, True), ref)
    with _in_place(lbm, nx, ny, rho0, walls=True, **CS) as lat:
        lat.step(165)
        ck = lat.checkpoint()
        lat.step(7)
        lat.restore(ck)
        lat.step(30)
        _same(_state(lbm, lat, True), ref)
