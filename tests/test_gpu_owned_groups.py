"""Owned builds tell how many cells the lane groups handed to the warp kernel: from 65,536 particles on those owned rows
that a full build hands over too, none below, where a list of the owned cells goes to the warp kernel.
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


@pytest.mark.parametrize("n", [65535, 65536])
def test_cells_handed_over_in_an_owned_build(n):
    L = 31.5
    pos = torch.from_numpy(inputs.clustered(n, L=L, seed=11)).cuda()
    box = ((0.0,) * 3, (L,) * 3, True)
    n_owned = 50000
    h = vt.vt_build_owned(pos, n_owned, None, *box)
    handed = vt.vt_status(h)["n_handed_over"]
    if n < 65536:
        assert handed == 0
    else:
        # the groups treat a cell the same whatever the other rows are
        full = vt.vt_status(vt.vt_build(pos, None, *box))["n_handed_over"]
        assert full - (n - n_owned) <= handed <= full and 0 < handed < n_owned
