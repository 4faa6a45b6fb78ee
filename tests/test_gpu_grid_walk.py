"""The nearest-particle grid against a brute-force argmin in FP64 (ties to the lower index): every node has to name the
same particle, also on a lattice whose nodes lie exactly on facets, edges and corners of the cells, at grid sizes around
the kernel's patch of 8 x 8 x 4 nodes, with sub-points, with three box lengths, and beside the walls of a box.  Each
particle's mass makes its density tell it from the others; a density is one division, so the comparison is exact.
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


def _nearest(x, box, periodic, G, S):
    axes = [(np.arange(G)[:, None] + (np.arange(S) + 0.5) / S).ravel() * (box[k] / G) for k in range(3)]
    q = np.stack(np.meshgrid(*axes, indexing="ij"), -1).reshape(-1, 3)
    out = np.empty(len(q), np.int64)
    for s in range(0, len(q), 4096):
        d = x[None, :, :] - q[s:s + 4096, None, :]
        if periodic:
            d = np.where(d > 0.5 * box, d - box, np.where(d < -0.5 * box, d + box, d))
        out[s:s + 4096] = np.argmin((d * d).sum(-1), axis=1)
    # (x, y, z, sub-points) -> nodes with x fastest, sub-points last
    return out.reshape(G, S, G, S, G, S).transpose(4, 2, 0, 5, 3, 1).reshape(G ** 3, S ** 3)


@pytest.mark.parametrize("kind,G,S,periodic,dtype", [
    ("uniform", 1, 1, True, np.float32), ("uniform", 7, 1, True, np.float32), ("uniform", 9, 1, False, np.float64),
    ("uniform", 33, 1, True, np.float64), ("uniform", 5, 2, False, np.float32), ("uniform", 3, 3, True, np.float32),
    ("clumps", 17, 1, True, np.float32), ("clumps", 16, 1, False, np.float32),
    ("lattice", 8, 1, True, np.float32), ("lattice", 16, 1, True, np.float64), ("lattice", 16, 1, False, np.float32)])
def test_every_node_finds_its_particle(kind, G, S, periodic, dtype):
    rng = np.random.default_rng(G * 10 + S)
    box = np.array([1.0, 1.0, 1.0]) if periodic else np.array([1.0, 0.5, 2.0])
    if kind == "lattice":
        x = np.stack(np.meshgrid(*[(np.arange(8) + 0.5) / 8] * 3, indexing="ij"), -1).reshape(-1, 3)
    elif kind == "clumps":
        x = np.where(rng.random((2000, 1)) < 0.5, rng.random((2000, 3)), 0.5 + 0.01 * rng.standard_normal((2000, 3)))
    else:
        x = rng.random((1500, 3))
    x = np.minimum((x * box).astype(dtype), np.nextafter(box.astype(dtype), dtype(0)))
    mass = (1.0 + rng.random(len(x))).astype(dtype)
    h = vt.vt_build(torch.from_numpy(x).cuda(), torch.from_numpy(mass).cuda(), (0.0,) * 3, tuple(box), periodic)
    dens = vt.density(h).double().cpu().numpy()
    got = vt.grid_density(h, G, S).double().cpu().numpy().reshape(-1)
    want = dens[_nearest(x.astype(np.float64), box, periodic, G, S)].mean(1)
    assert np.abs(got / want - 1).max() <= (0.0 if S == 1 else 1e-6)
