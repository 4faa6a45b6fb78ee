"""The Green-Gauss gradient of FP32 sets, whose quotients area / distance are formed from pairs of floats, against the
same particles as an FP64 set, whose quotients are FP64: boxes scaled by powers of two change no bit of the geometry, so
that the difference is the FP32 rounding of results (2^-24) and of the facet records of either set (a few 2^-24 of
the largest gradient; 1e-6 allowed)."""
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


@pytest.mark.parametrize("n,periodic,exponent", [(2000, True, 0), (2000, True, -12), (2000, True, 7), (33, False, 0)])
def test_fp32_results_match_fp64_quotients(n, periodic, exponent):
    x = inputs.uniform(n, seed=n, dtype=np.float32) * np.float32(2.0 ** exponent)
    box = (float(2.0 ** exponent),) * 3
    g = [vt.gradient_gg(vt.vt_build(torch.from_numpy(x.astype(dt)).cuda(), None, (0.0,) * 3, box, periodic)).double().cpu().numpy()
         for dt in (np.float32, np.float64)]
    assert np.isfinite(g[0]).all()
    assert np.abs(g[0] - g[1]).max() <= 1e-6 * np.abs(g[1]).max()
