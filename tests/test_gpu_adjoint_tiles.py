"""The tiled reverse step at the edges of its tiles (32 columns, 4 to 16 rows):
remainders of one row or column, channels as low as one tile's halo, wetting
ghosts, tau != 1, periodic and pressure-column ends, against central
differences of the FP64 oracle along a random direction of rho0.

Supercritical fluid: no phase weight, so J is smooth. The central difference at
h = 1e-5 has truncation error O(h^2) ~ 1e-10 and rounding error about
1e-16 J / h ~ 1e-10 of the sum of |g v|; 1e-6 of it is asked for. The FP32
reverse sweep rounds each of some 50 operations per step to 6e-8: its gradient
of J_p (whose terms have one sign; J_tau's nearly cancel on the smallest grids)
is asked to be within 1e-4 of the FP64 one in the 2-norm.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

# nx, ny, pressure columns, wetting, tau, steps
GRIDS = [(33, 18, True, 0.0, 1.0, 12), (64, 34, True, 0.002, 1.0, 12), (35, 5, True, 0.003, 1.0, 9),
         (31, 4, True, 0.0, 1.1, 9), (4, 19, True, 0.001, 1.0, 7), (97, 19, False, 0.003, 1.2, 12),
         (5, 6, False, 0.0, 1.0, 7), (161, 67, True, 0.0, 0.9, 10), (32, 130, False, 0.0, 1.0, 8)]


@pytest.mark.parametrize("nx,ny,bc_x,wet,tau,steps", GRIDS)
def test_gradient_along_a_direction_matches_the_oracle(orc, nx, ny, bc_x, wet, tau, steps):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    from paper_2103_08301_gb300.adjoint import Adjoint
    T, kappa, dp = 1.1, 0.5, 2e-4
    s0 = orc.Setup(nx=nx, ny=ny, walls=True, bc_x=False, T_over_Tc=T, kappa=kappa)
    p_ref = orc.cs_p0(s0.a, s0.b, s0.R, s0.T, 0.13)
    s = orc.Setup(nx=nx, ny=ny, walls=True, bc_x=bc_x, T_over_Tc=T, kappa=kappa, dp=dp, p_ref=p_ref, tau=tau,
                  wet=wet)
    rho0 = synth.airway_rho0(nx, ny, max(1, ny // 6), nx // 3, max(2, nx // 5), 0.15, 0.12, noise=1e-3, seed=4)
    v = np.random.RandomState(nx).standard_normal((ny, nx))

    def J(r):
        _, d = orc.run(s, orc.init(s, r), steps)
        return np.array([d["J"], d["Jp"]])

    h = 1e-5
    fd = (J(rho0 + h * v) - J(rho0 - h * v)) / (2 * h)
    grads = {}
    for reverse in (64, 32):
        with Adjoint(nx, ny, steps, walls=True, bc_x=bc_x, T_over_Tc=T, kappa=kappa, p_ref=p_ref, tau=tau, wetting=wet,
                     precision=64, reverse_precision=reverse, block_steps=5) as adj:
            adj.forward(rho0, dp=dp)
            grads[reverse] = [adj.backward(1.0, 0.0)[0], adj.backward(0.0, 1.0)[0]]
    for k in range(2):
        g = grads[64][k]
        assert abs((g * v).sum() - fd[k]) <= 1e-6 * np.abs(g * v).sum(), (k, (g * v).sum(), fd[k])
    assert np.linalg.norm(grads[32][1] - grads[64][1]) <= 1e-4 * np.linalg.norm(grads[64][1])
