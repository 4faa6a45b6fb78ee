"""Volumes at the sizes where the sort changes: one run, a run and a remainder, many runs, and the largest set sorted in
runs with its neighbours on both sides.  A key lost or doubled by the sort loses a cell: volumes are compared one by one
with the FP64 oracle (within 2e-5) and, for the large sets, with those of the same points in another order (twice that);
they add up to the box.  Half of the points lie in clumps narrower than the spacing of the Morton keys, so that many
keys are equal; clumps that narrow are beyond the FP32 filter's search, hence the FP64 clipping.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1601_06429_gb300 import binding as vt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1601_06429_gb300.build import build

    build()
    vt.load_library()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _points(n, seed):
    rng = np.random.default_rng(seed)
    centre = rng.random((max(1, n // 64), 3)) * 0.9 + 0.05
    clump = centre[rng.integers(len(centre), size=n)] + 1e-6 * rng.standard_normal((n, 3))
    x = np.where(rng.random((n, 1)) < 0.5, clump, rng.random((n, 3)))
    return np.unique(x, axis=0)[rng.permutation(n)] if n > 1 else x


def _volumes(x):
    h = vt.vt_build(torch.from_numpy(x).cuda(), None, (0.0,) * 3, (1.0,) * 3, False, "plain64")
    return vt.cells(h)[0].double().cpu().numpy()


@pytest.mark.parametrize("n", [1, 2, 31, 33, 1023, 1024, 1025, 2047, 2049])
def test_volumes_against_the_oracle(n, oracle_mod):
    x = _points(n, n)
    o = oracle_mod.cells(x, 0.0, 1.0, False, mode="certified" if n > 100 else "brute")
    v = _volumes(x)
    assert np.abs(v / o["vol"] - 1).max() <= 2e-5


@pytest.mark.parametrize("n", [32768, 65535, 65536, 65537])
def test_volumes_of_another_order(n):
    x = _points(n, n)
    order = np.random.default_rng(1).permutation(n)
    v, w = _volumes(x), _volumes(x[order])
    assert np.abs(w / v[order] - 1).max() <= 4e-5
    assert abs(v.sum() - 1) <= 2e-5
