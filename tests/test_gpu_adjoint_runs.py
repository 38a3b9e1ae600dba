"""Blocks of states whose fields do not fit one buffer (256 MiB) are walked in
several runs, prepared beside the chain: the gradients are those of shorter blocks
that need no split, bit for bit (the same states, the same chain of steps).
512 x 512: a state's fields take 24 MiB, so a buffer holds ten.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reverse", [64, 32])
def test_gradient_does_not_depend_on_how_blocks_are_walked(orc, reverse):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    from paper_2103_08301_gb300.adjoint import Adjoint
    nx, ny, steps = 512, 512, 46
    g, l, _ = orc.Setup(nx=nx, ny=ny, walls=True, bc_x=True, T_over_Tc=0.85, kappa=0.5).coexistence()
    rho0 = synth.airway_rho0(nx, ny, 24, 128, 64, l, g, noise=1e-3, seed=9)
    out = []
    for block in (46, 23, 7):  # five runs; three and three; one a block, the last block shorter
        with Adjoint(nx, ny, steps, T_over_Tc=0.85, kappa=0.5, precision=32, reverse_precision=reverse,
                     block_steps=block) as adj:
            J = adj.forward(rho0, dp=2e-4)
            first = adj.backward(1.0, 0.5)
            again = adj.backward(1.0, 0.5)  # from the states that the first pass left
            assert np.array_equal(first[0].view(np.uint64), again[0].view(np.uint64)) and first[1] == again[1]
            out.append((J, first))
    for J, (grad, drive) in out[1:]:
        assert np.array_equal(grad.view(np.uint64), out[0][1][0].view(np.uint64))
        assert drive == out[0][1][1]
        # sums over the states, taken block by block: FP64 rounding of up to 46 terms a column
        assert all(abs(a - b) <= 1e-13 * abs(b) for a, b in zip(J, out[0][0]))
