"""The volume-averaged grid where facets meet within rounding of one point: lattices displaced by 1e-7 to 1e-4 of the
box, whose side tests contradict each other in FP32, against the FP64 oracle; and cells of many facets, whose parts of a
voxel outgrow the 40 planes of a lane group.  No part may be lost, and the tolerance is that of the other voxel tests
(2e-5 of the largest voxel).
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


def lattice(kind, shift, seed):
    if kind == "sc":
        x = inputs.sc_lattice(12)
    elif kind == "bcc":
        x = inputs.bcc_lattice(9)
    else:  # face-centred cubic: cube corners and face centres
        g1 = (np.arange(8) + 0.25) / 8.0
        a = np.stack(np.meshgrid(g1, g1, g1, indexing="ij"), -1).reshape(-1, 3)
        x = np.concatenate([a] + [a + np.array(o) / 16.0 for o in ((0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1))][1:])
    x = x + inputs.rng(seed).uniform(-shift, shift, x.shape)
    return (x - np.floor(x)).astype(np.float32)


def check(x, G, periodic, precision, oracle_mod):
    x64 = x.astype(np.float64)
    o = oracle_mod.cells(x64, 0.0, 1.0, periodic, mode="certified", face_cap=400)
    ref = oracle_mod.grid_volume_density(x64, 1.0 / o["vol"], 0.0, 1.0, G, periodic=periodic)
    h = vt.vt_build(torch.from_numpy(x).cuda(), None, (0.0,) * 3, (1.0,) * 3, periodic, precision)
    got = vt.grid_density_volume(h, G).double().cpu().numpy()
    assert vt.vt_status(h)["n_grid_failed"] == 0
    assert np.abs(got - ref).max() <= 2e-5 * ref.max()


@pytest.mark.parametrize("G", [8, 16, 32])
@pytest.mark.parametrize("kind,shift", [("fcc", 1e-7), ("fcc", 1e-6), ("fcc", 1e-5), ("fcc", 1e-4), ("sc", 1e-6),
                                        ("sc", 1e-5), ("bcc", 1e-6)])
def test_lattices_close_to_degenerate(kind, shift, G, oracle_mod):
    check(lattice(kind, shift, seed=G), G, True, "plain64", oracle_mod)


def sphere(facets):
    """A particle inside a sphere of others, whose cell has that many facets."""
    g = inputs.rng(facets)
    k = np.arange(facets)
    z, phi = 1.0 - (2.0 * k + 1.0) / facets, k * (np.pi * (3.0 - np.sqrt(5.0)))
    s = np.stack([np.sqrt(1.0 - z * z) * np.cos(phi), np.sqrt(1.0 - z * z) * np.sin(phi), z], 1)
    return np.concatenate([[[0.5, 0.5, 0.5]], 0.5 + (0.36 + 1e-4 * g.random((facets, 1))) * s]).astype(np.float32)


@pytest.mark.parametrize("facets", [30, 60, 110])
@pytest.mark.parametrize("G", [2, 3, 7])
def test_cells_of_many_facets(facets, G, oracle_mod):
    """At G = 3 the middle voxel takes nearly all of the facets."""
    check(sphere(facets), G, False, "filter32", oracle_mod)


def test_parts_beyond_the_larger_polytope_are_counted():
    """200 facets, of which the middle voxel of 3 holds some 150 (130 fit); the same handle then fills 7^3 voxels."""
    x = sphere(200)
    h = vt.vt_build(torch.from_numpy(x).cuda(), None, (0.0,) * 3, (1.0,) * 3, False)
    vt.grid_density_volume(h, 3)
    assert vt.vt_status(h)["n_grid_failed"] == 1
    got = vt.grid_density_volume(h, 7).double()
    assert vt.vt_status(h)["n_grid_failed"] == 0
    assert abs(float(got.mean()) - len(x)) <= 1e-5 * len(x)  # every particle has mass 1
