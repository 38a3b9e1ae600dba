"""Where lbm_fields writes: device destinations that hold the output are written by
the kernel; one whose allocation is too short is refused by the copy that host
destinations take, with an error status, and the context goes on.
"""
import ctypes as C

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [32, 64])
def test_short_device_destination_is_refused(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    import paper_2103_08301_gb300 as lbm
    nx, ny = 512, 640 * 32 // precision  # 1.25 MiB a field
    cuda = lbm.lib()  # the runtime it is linked with answers to the same handle
    rho0 = synth.airway_rho0(nx, ny, ny // 16, nx // 4, nx // 8, 0.2759, 0.02185)
    with lbm.Lattice(nx, ny, rho0, precision=precision, walls=True, bc_x=True, T_over_Tc=0.85, kappa=0.5, dp=1e-3) as lat:
        lat.step(3)
        want = lat.fields()["rho"]
        short = C.c_void_p()
        assert cuda.cudaMalloc(C.byref(short), C.c_size_t(1 << 20)) == 0  # allocations start on 2 MiB of memory
        try:
            assert cuda.lbm_fields(lat.ctx, short, None, None, None, None) == lbm.LBM_ERR_CUDA
            assert cuda.cudaGetLastError() == 1  # cudaErrorInvalidValue, kept by the runtime until it is read
        finally:
            assert cuda.cudaFree(short) == 0
        lat.step(0)  # the context is still in order
        whole = torch.full((2, ny, nx), -1.0, dtype=torch.float32 if precision == 32 else torch.float64, device="cuda")
        lat.fields_into(rho=whole[0])
        assert np.array_equal(whole[0].cpu().numpy(), want)
        assert bool((whole[1] == -1.0).all())


@pytest.mark.parametrize("precision", [32, 64])
def test_masked_fields_alike_in_every_destination(precision):
    """All outputs, one output, device and host memory: the same values, solid
    nodes zero, whatever the scratch held before."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08301_gb300 import build
    build.build()
    import paper_2103_08301_gb300 as lbm
    nx, ny = 203, 61
    dt = torch.float32 if precision == 32 else torch.float64
    mask = np.zeros((ny, nx), np.uint8)
    mask[20:30, 60:75] = mask[1:9, 120:130] = 1
    rho0 = synth.airway_rho0(nx, ny, 4, 30, 20, 0.2759, 0.02185)
    shapes = {"rho": (ny, nx), "vx": (ny, nx), "vy": (ny, nx), "tau_wall": (2, nx), "p_wall": (2, nx)}
    with lbm.Lattice(nx, ny, rho0, precision=precision, walls=True, bc_x=True, T_over_Tc=0.85, kappa=0.5, dp=1e-3,
                     mask=mask) as lat:
        lat.step(20)
        dev = {k: torch.full(s, 7.0, dtype=dt, device="cuda") for k, s in shapes.items()}
        lat.fields_into(**dev)
        host = lat.fields()
        assert (host["rho"][mask == 1] == 0).all()
        for k, s in shapes.items():
            assert np.array_equal(dev[k].cpu().numpy(), host[k]), k
            one = torch.full(s, 7.0, dtype=dt, device="cuda")
            lat.fields_into(**{k: one})
            assert np.array_equal(one.cpu().numpy(), host[k]), k
            one = np.full(s, 7.0, lat.dtype)
            lat.fields_into(**{k: one})
            assert np.array_equal(one, host[k]), k
        mixed = np.full((ny, nx), 7.0, lat.dtype)
        lat.fields_into(rho=dev["vx"], vx=mixed)
        assert np.array_equal(dev["vx"].cpu().numpy(), host["rho"]) and np.array_equal(mixed, host["vx"])
