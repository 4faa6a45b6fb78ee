"""Searches of the lane-group kernels that outgrow a cell's list of 96 candidates: the list is read back by all lanes of
the warp and shortened, in the middle of a leaf's points.  A k_target of 120 starts from 1.6 times the distance of the 30th
mate, a ball of about 120 points, so that nearly every cell's first pass overflows.  The warp kernel (256 candidates)
gives the bits to compare with.
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


@pytest.mark.parametrize("lanes", [4, 8])
@pytest.mark.parametrize("kind,n,dtype,periodic", [("uniform", 4097, np.float64, False), ("uniform", 20011, np.float32, True),
                                                   ("clustered", 20011, np.float32, True)])
def test_overflowing_lists_give_the_same_cells(kind, n, dtype, periodic, lanes):
    L = 1.0 if kind == "uniform" else float(np.float32(100.0 * (n / 2097152.0) ** (1.0 / 3.0)))
    x = inputs.uniform(n, seed=n, L=L, dtype=np.float32) if kind == "uniform" else inputs.clustered(n, L=L, seed=n)
    pos = torch.from_numpy(x.astype(dtype)).cuda()
    out = []
    for tpc in (32, lanes):
        h = vt.vt_build(pos, None, (0.0,) * 3, (L,) * 3, periodic, k_target=120, threads_per_cell=tpc)
        out.append(vt.cells(h) + (vt.gradient(h), vt.cell_radius(h)))
    assert all(torch.equal(a, b) for a, b in zip(*out))
