"""lbm_launch_info describes one kernel: tiles where the step runs by tiles, the
general-geometry kernels where nodes are solid.
"""
import numpy as np
import pytest

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


@pytest.mark.parametrize("nx,ny,walls,precision", [(128, 128, False, 64), (4096, 512, True, 64), (512, 128, True, 32),
                                                   (1500, 202, True, 32)])
def test_tiles(lbm, nx, ny, walls, precision):
    with lbm.Lattice(nx, ny, np.full((ny, nx), 0.1), precision=precision, walls=walls, T_over_Tc=1.1) as lat:
        info = lat.launch_info()
    rows, th = ny - 2 * walls, info["threads"] // 32
    assert info["threads"] == 32 * th and 2 <= th <= 8
    assert info["units"] == -(-nx // 32) * -(-rows // th) and info["ctas"] <= info["units"]
    assert info["staged"]


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("nx,ny", [(256, 64), (1024, 512)])
def test_solid_nodes(lbm, nx, ny, precision):
    import torch
    mask = np.zeros((ny, nx), np.uint8)
    mask[ny // 2, nx // 2] = 1
    with lbm.Lattice(nx, ny, np.full((ny, nx), 0.1), precision=precision, walls=True, T_over_Tc=1.1, mask=mask) as lat:
        info = lat.launch_info()
    most = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    assert info == {"ctas": min(nx * ny // 256, most), "threads": 256, "units": nx * ny, "staged": False}
