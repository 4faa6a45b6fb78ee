"""Sheets of particles between far walls: cells as long as the box, whose neighbours all lie within the balls of their
vertices, so that the warp kernel's searches against those balls leave nothing out and are given up.  The five cells with most
candidates of the 70,000 (up to 58,000) and some others against the FP64 oracle; and the balls may not cost a multiple of
what the cells do without them (105 ms; 412 ms with the balls in every search).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1601_06429_gb300 import binding as vt
from paper_1601_06429_gb300 import inputs

pytestmark = pytest.mark.gpu
WIDE = [21855, 35398, 34216, 2137, 61682]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1601_06429_gb300.build import build

    build()
    vt.load_library()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.fixture(scope="module")
def sheet():
    x = inputs.rng(3).random((70000, 3))
    x[:, 2] = 0.5 + 1e-3 * x[:, 2]
    return x.astype(np.float32)


@pytest.mark.parametrize("precision,tpc,tol", [("filter32", 32, 2e-5), ("filter32", 0, 2e-5), ("plain64", 0, 1e-6)])
def test_cells_of_a_sheet_match_the_oracle(sheet, precision, tpc, tol, oracle_mod):
    h = vt.vt_build(torch.from_numpy(sheet).cuda(), None, (0.0,) * 3, (1.0,) * 3, False, precision, threads_per_cell=tpc)
    vol, off, ids = (t.cpu().numpy() for t in vt.cells(h))
    which = np.array(WIDE + inputs.rng(4).choice(len(sheet), 24, replace=False).tolist())
    o = oracle_mod.cells(sheet.astype(np.float64), 0.0, 1.0, False, which=which, mode="certified")
    ooff, oids = oracle_mod.neighbours(o)
    for k, i in enumerate(which):
        assert np.array_equal(ids[off[i]:off[i + 1]], oids[ooff[k]:ooff[k + 1]])
        assert abs(vol[i] - o["vol"][k]) <= tol * o["vol"][k]


@pytest.mark.parametrize("tpc", [32, 0])
def test_the_balls_do_not_multiply_the_time_of_a_sheet(sheet, tpc):
    pos = torch.from_numpy(sheet).cuda()
    ms = [vt.vt_status(vt.vt_build(pos, None, (0.0,) * 3, (1.0,) * 3, False, threads_per_cell=tpc))["t_clip_ms"] for _ in range(3)]
    assert min(ms) <= 210.0
