"""Owned builds tell how many cells the lane groups handed to the warp kernel: from 40,000 owned rows on those that a
full build hands over too, none below, however many particles there are, where a list of the owned cells goes to the warp
kernel.
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


@pytest.mark.parametrize("n_owned", [1, 3000, 39999, 40000])
def test_cells_handed_over_in_an_owned_build(n_owned):
    n, L = 100000, 36.25
    pos = torch.from_numpy(inputs.clustered(n, L=L, seed=11)).cuda()
    box = ((0.0,) * 3, (L,) * 3, True)
    h = vt.vt_build_owned(pos, n_owned, None, *box)
    handed = vt.vt_status(h)["n_handed_over"]
    full = vt.vt_build(pos, None, *box)
    if n_owned < 40000:
        assert handed == 0
    else:
        # the groups treat a cell the same whatever the other rows are
        most = vt.vt_status(full)["n_handed_over"]
        assert most - (n - n_owned) <= handed <= most and 0 < handed < n_owned
    assert torch.equal(vt.cells(h)[0][:n_owned], vt.cells(full)[0][:n_owned])
