"""The FP32 reverse step on the one channel height (fluid rows = 1 mod 720720) for
which every tile height leaves a single row over, so that the two rows next to
the top wall lie in two tiles. Against the FP64 reverse sweep: three steps round
each of some 50 operations to 6e-8, so the gradient of J_p (whose terms have one
sign) next to either wall is asked to be within 1e-4 in the 2-norm.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_single_row_left_over_at_the_top_wall(orc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    from paper_2103_08301_gb300.adjoint import Adjoint
    nx, ny = 4, 720723
    s0 = orc.Setup(nx=8, ny=8, walls=True, bc_x=False, T_over_Tc=1.1, kappa=0.5)
    p_ref = orc.cs_p0(s0.a, s0.b, s0.R, s0.T, 0.13)
    rho0 = 0.13 * (1 + 1e-3 * np.random.RandomState(1).standard_normal((ny, nx)))
    grads = {}
    for reverse in (64, 32):
        with Adjoint(nx, ny, 3, walls=True, bc_x=True, T_over_Tc=1.1, kappa=0.5, p_ref=p_ref, precision=32,
                     reverse_precision=reverse) as adj:
            adj.forward(rho0, dp=2e-4)
            grads[reverse] = adj.backward(0.0, 1.0)[0]
    for rows in (slice(0, 14), slice(ny - 14, ny)):
        g64, g32 = grads[64][rows], grads[32][rows]
        assert np.linalg.norm(g32 - g64) <= 1e-4 * np.linalg.norm(g64), rows
