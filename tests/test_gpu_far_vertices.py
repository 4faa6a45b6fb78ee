"""FP64 geometry of cells whose vertices lie thousands of search radii away: the first particles found are 1e-6 to 1e-4
of the box off, the vertices on the box wall.  A particle that cuts just one far vertex off, by some 1e-9 of the squared
box side, is a neighbour the search must not leave out.  Compared with the FP64 oracle's facets.
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


def narrow_cell(seed):
    """Site 0, four particles around it that leave it a cone up to the wall x = 1, eight behind it, and one more whose
    plane passes a corner of the cone's base at a relative depth of 1e-9 to 1e-8."""
    g = inputs.rng(seed)
    site = np.full(3, 0.5)
    ray = [np.array([0.5, sy * 0.3 * g.uniform(0.7, 1.3), sz * 0.3 * g.uniform(0.7, 1.3)])
           for sy, sz in ((1, 1), (-1, 1), (-1, -1), (1, -1))]
    rho = g.uniform(1e-4, 2e-4)
    delta = rho / 50.0
    cone = []
    for k in range(4):
        n = np.cross(ray[k], ray[(k + 1) % 4])
        n *= np.sign(-n[0]) / np.linalg.norm(n)  # outward: away from the axis of the cone
        cone.append(n)
    x = np.concatenate([[site], site + delta * np.array(cone)])
    d = x[1:5] - x[0]
    # the corner on planes 3 and 0 (both hold ray 0) and the wall
    v = np.linalg.solve(np.stack([2.0 * d[3], 2.0 * d[0], [1.0, 0.0, 0.0]]), [d[3] @ d[3], d[0] @ d[0], 0.5])
    out = np.array([-(v[1] / abs(v[1]) * v[1] + v[2] / abs(v[2]) * v[2]) / v[0], np.sign(v[1]), np.sign(v[2])])
    out /= np.linalg.norm(out)
    b = 10.0 ** g.uniform(-8.7, -7.9)
    s = (b + rho * rho) / (2.0 * rho * np.linalg.norm(v))
    p = rho * (np.sqrt(1.0 - s * s) * out + s * v / np.linalg.norm(v))
    back = delta * (np.array([-1.5, 0.0, 0.0]) + 0.5 * g.uniform(-1.0, 1.0, (8, 3)))
    return np.concatenate([x, site + back, [site + p]])


def test_a_particle_that_cuts_one_far_vertex_is_a_neighbour(oracle_mod):
    lost = []
    for seed in range(96):
        x = narrow_cell(seed)
        h = vt.vt_build_owned(torch.from_numpy(x).cuda(), 1, None, (0.0,) * 3, (1.0,) * 3, False, "plain64")
        _, off, ids = (t.cpu().numpy() for t in vt.cells(h))
        o = oracle_mod.cells(x, 0.0, 1.0, False, which=[0], mode="certified")
        ref = oracle_mod.neighbours(o)[1]
        assert len(x) - 1 in ref
        if not np.array_equal(ids[:off[1]], ref):
            lost.append(seed)
    assert not lost
