"""Wide cells beside a dense halo: their searches test nodes and points against the balls of the cell's vertices (from
8193 particles on), which has to leave out only what cannot cut.  Compared with the FP64 oracle.
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


@pytest.mark.parametrize("n", [8192, 8193])
@pytest.mark.parametrize("precision,tol", [("filter32", 2e-5), ("plain64", 1e-6)])
def test_a_void_beside_a_dense_halo_matches_the_oracle(n, precision, tol, oracle_mod):
    """Most points in one small halo, a few around it: the few bound wide cells that face thousands of halo points."""
    g = inputs.rng(31)
    halo = 0.5 + 0.02 * g.normal(size=(n - 60, 3))
    x = np.concatenate([halo, g.random((60, 3))]).clip(0.0, 1.0).astype(np.float32)
    h = vt.vt_build(torch.from_numpy(x).cuda(), None, (0.0,) * 3, (1.0,) * 3, False, precision)
    vol, off, ids = (t.cpu().numpy() for t in vt.cells(h))
    o = oracle_mod.cells(x.astype(np.float64), 0.0, 1.0, False, mode="certified")
    ooff, oids = oracle_mod.neighbours(o)
    assert np.array_equal(off, ooff) and np.array_equal(ids, oids)
    assert (np.abs(vol - o["vol"]) / o["vol"]).max() <= tol
