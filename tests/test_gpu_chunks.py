"""Lane groups over more than one chunk of their memory (2,097,152 cells) in batched and owned builds, against the warp
kernel bit for bit: sets that end, begin and lie across the edge of a chunk, and owned rows on both sides of it.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1601_06429_gb300 import binding as vt
from paper_1601_06429_gb300 import inputs

pytestmark = pytest.mark.gpu
CHUNK = 2097152


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1601_06429_gb300.build import build

    build()
    vt.load_library()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def same(a, b):
    return all(torch.equal(p, q) for p, q in zip(vt.cells(a), vt.cells(b))) and torch.equal(vt.cell_radius(a), vt.cell_radius(b))


@pytest.mark.parametrize("edge", [0, -13, 1000])
def test_sets_around_the_edge_of_a_chunk(edge):
    off = np.array([0, 1500000, CHUNK + edge, CHUNK + edge + 40, CHUNK + 90000], np.int64)
    pos = torch.from_numpy(inputs.uniform(int(off[-1]), seed=8, dtype=np.float32)).cuda()
    boxes = np.tile([0.0, 0.0, 0.0, 1.0, 1.0, 1.0], (4, 1))
    a, b = (vt.vt_build_batched(pos, off, boxes, threads_per_cell=t) for t in (0, 32))
    assert same(a, b)


def test_owned_rows_on_both_sides_of_the_edge_of_a_chunk():
    n, n_owned = CHUNK + 70001, 1200000
    pos = torch.from_numpy(inputs.uniform(n, seed=9, dtype=np.float32)).cuda()
    full = vt.vt_build(pos, None, threads_per_cell=32)
    part = vt.vt_build_owned(pos, n_owned, None)
    assert 0 < vt.vt_status(part)["n_handed_over"] < n_owned // 20
    for a, b in ((vt.cells(full)[0], vt.cells(part)[0]), (vt.cell_radius(full), vt.cell_radius(part))):
        assert torch.equal(a[:n_owned], b[:n_owned]) and not b[n_owned:].any()
    vt.vt_rebuild(part, pos)
    assert torch.equal(vt.cells(part)[0][:n_owned], vt.cells(full)[0][:n_owned])
