"""A checkpoint taken under one launch plan and restored under another with
fewer CTAs: the diagnostic totals are those of the checkpoint, and go on from
there. The partials are added in another order: sums of at most 8192 FP64
partials of both signs round to 1e-12 of the sum of their sizes.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("ctas", [(5, 1), (1, 5)])
def test_totals_survive_another_plan(orc, precision, ctas):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    import paper_2103_08301_gb300 as lbm
    nx, ny = 1024, 256
    kw = dict(walls=True, bc_x=True, T_over_Tc=0.85, kappa=0.5, dp=1e-3)
    g, l, _ = orc.Setup(nx=nx, ny=ny, **kw).coexistence()
    rho0 = synth.airway_rho0(nx, ny, 12, 256, 64, l, g)
    with lbm.Lattice(nx, ny, rho0, precision=precision, **kw) as a, \
            lbm.Lattice(nx, ny, rho0, precision=precision, **kw) as b:
        a.set_option(lbm.LBM_OPT_CTAS_PER_SM, ctas[0])
        b.set_option(lbm.LBM_OPT_CTAS_PER_SM, ctas[1])
        a.step(60)
        b.restore(a.checkpoint())
        for _ in range(2):
            da, db = a.diag(), b.diag()
            size = da["step"] * 2 * nx * max(abs(da["tau_wall_min"]), abs(da["tau_wall_max"]))
            assert abs(db["wall_shear_sum"] - da["wall_shear_sum"]) <= 1e-12 * size
            # FP32 plans add up to 16 rows of a lane in FP32 first
            assert abs(db["mass"] / da["mass"] - 1) <= (1e-12 if precision == 64 else 1e-6)
            for k in ("tau_wall_min", "tau_wall_max", "p_wall_min", "p_wall_max", "nan_detected", "step"):
                assert da[k] == db[k], k
            a.step(20)
            b.step(20)
