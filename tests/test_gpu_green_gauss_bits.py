"""The Green-Gauss gradient of FP32 results is formed as accurately as that of FP64 results: the same particles as an FP32
and as an FP64 set have the same cells, facet records and densities, and the quotients area / distance agree to a few units
of 2^-53.  A simple cubic lattice displaced by 1e-3 of its spacing, with masses 1 and 2 in turn: a gradient's terms are a
thousand times their sum.  Rounded to FP32 the gradients of the two sets differ where one lies within the difference of a
rounding boundary, which for 98,304 values and a difference of 2^-53 of the terms is 98,304 x 2 x 1000 x 2^-53 / 2^-24 =
0.4 values: three are allowed.
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


@pytest.mark.parametrize("precision", ["filter32", "plain64"])
def test_gradients_of_fp32_and_fp64_sets_round_to_the_same(precision):
    n = 32
    x = torch.from_numpy(inputs.sc_lattice(n, perturb=1e-3 / n, seed=3, dtype=np.float32)).cuda()
    mass = torch.from_numpy(1.0 + (np.indices((n, n, n)).sum(0).reshape(-1) & 1)).cuda()
    h = [vt.vt_build(p, mass, (0.0,) * 3, (1.0,) * 3, True, precision) for p in (x, x.double())]
    assert torch.equal(vt.density(h[0]), vt.density(h[1]).float())
    g = [vt.gradient_gg(k) for k in h]
    assert int((g[0] != g[1].float()).sum()) <= 3
