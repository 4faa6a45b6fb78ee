"""The volume-averaged grid and the weighted centroidal gradient at the sizes where their kernels change paths, against
the FP64 oracle: cells inside one voxel, cells over a few voxels, cells over more voxels than a warp walks alone, voxels
inside one cell, voxels across the faces of a periodic box; facets with more corners than a lane's polygon holds, and
facets cut by box walls.  Tolerances are those of the parity tests (2e-5 of the largest voxel; 1e-4 of a particle's
gradient plus 1e-5 of the largest).
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
    (300, 64, True, np.float32),      # every cell over more voxels than one unit of work, the units not full
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


def ring(corners, seed):
    """Two sites whose common facet has `corners` corners: on the axis of a ring of sites, and a few far ones."""
    g = inputs.rng(seed)
    a = 2.0 * np.pi * (np.arange(corners) + 0.1 * g.random(corners)) / corners
    rr = 0.3 + 1e-4 * g.random(corners)
    c = np.stack([0.5 + rr * np.cos(a), 0.5 + rr * np.sin(a), 0.5 + 1e-4 * g.random(corners)], 1)
    poles = np.array([[0.5, 0.5, 0.48], [0.5, 0.5, 0.52]])
    return np.concatenate([poles, c, g.random((20, 3)) * np.array([1.0, 1.0, 0.05])])


@pytest.mark.parametrize("points,periodic", [("ring10", False), ("ring22", False), ("ring40", False), ("few", False),
                                             ("uniform", True), ("halo", False)])
def test_weighted_gradient(points, periodic, oracle_mod):
    if points.startswith("ring"):
        x = ring(int(points[4:]), seed=5)
    elif points == "few":
        x = inputs.uniform(9, seed=2)
    elif points == "halo":
        x = (inputs.halo_sets(n_sets=1, nmin=2000, nmax=2001, seed=8)[0].astype(np.float64) + 1.0) / 2.0
    else:
        x = inputs.uniform(1001, seed=3)
    w = np.random.default_rng(4).random(len(x)) + 0.5
    o = oracle_mod.cells(x, 0.0, 1.0, periodic, mode="certified")
    ref = oracle_mod.cvt_weighted_gradient(o, x, w)
    h = vt.vt_build(torch.from_numpy(x).cuda(), None, (0.0,) * 3, (1.0,) * 3, periodic, "plain64")
    got = vt.backward_weighted(h, torch.from_numpy(w)).cpu().numpy()
    assert vt.vt_status(h)["n_grid_failed"] == 0
    scale = np.linalg.norm(ref, axis=1)
    assert (np.linalg.norm(got - ref, axis=1) <= 1e-4 * scale + 1e-5 * scale.max()).all()
