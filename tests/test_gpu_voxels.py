"""The volume-averaged grid at the sizes where its kernel changes paths, against the FP64 oracle: cells inside one voxel,
cells over a few voxels, cells over more voxels than a warp walks alone, voxels inside one cell, voxels across the faces
of a periodic box.  The tolerance is that of the parity tests (2e-5 of the largest voxel).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1601_06429_gb300 import binding as vt
from paper_1601_06429_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1601_06429_gb300.build import build

    build()
    vt.load_library()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("n,G,periodic,dtype", [
    (12, 40, False, np.float64),      # a cell covers thousands of voxels
    (300, 13, True, np.float32), (300, 1, True, np.float32),
    (2500, 37, False, np.float32), (2500, 2, True, np.float64),
    (9000, 5, True, np.float32)])
def test_voxel_averages(n, G, periodic, dtype, oracle_mod):
    x = inputs.uniform(n, seed=n + G, dtype=np.float32).astype(dtype)
    x64 = x.astype(np.float64)
    o = oracle_mod.cells(x64, 0.0, 1.0, periodic, mode="certified")
    ref = oracle_mod.grid_volume_density(x64, 1.0 / o["vol"], 0.0, 1.0, G, periodic=periodic)
    h = vt.vt_build(torch.from_numpy(x).cuda(), None, (0.0,) * 3, (1.0,) * 3, periodic)
    got = vt.grid_density_volume(h, G).double().cpu().numpy()
    assert vt.vt_status(h)["n_grid_failed"] == 0
    assert np.abs(got - ref).max() <= 2e-5 * ref.max()
    # again on the same handle (the lists and the accumulator are cleared)
    assert np.abs(vt.grid_density_volume(h, G).double().cpu().numpy() - got).max() <= 1e-6 * ref.max()
