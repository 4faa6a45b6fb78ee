"""The lane-group kernels (4 or 8 lanes per cell; the library's choice from 65,536 particles on) against the warp kernel.

Both cut a cell with the same planes in the same order and sum its facets in the same order, so every output has to be
the same bits, whatever the group size and whichever cells share a warp.  The warp kernel is compared with the FP64
oracle in test_gpu_parity.  Sizes: one bucket of the search tree and its edges, the library's threshold, a chunk of the kernels' memory
(2,097,152 cells) and its edge, uneven sets that share a bucket, owned rows.
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


def outputs(h):
    vol, off, ids = vt.cells(h)
    cen, energy = vt.moments(h)
    w = torch.linspace(0.0, 1.0, h.N, device="cuda", dtype=h.dtype)
    return dict(vol=vol, off=off, ids=ids, dens=vt.density(h), grad=vt.gradient(h), gg=vt.gradient_gg(h), cen=cen,
                energy=energy, rad=vt.cell_radius(h), adjoint=vt.backward(h, w, 0.5))


def same(a, b):
    for k in a:
        assert torch.equal(a[k], b[k]), k


def points(kind, n, dtype, L):
    if kind == "uniform":
        return inputs.uniform(n, seed=n, L=L, dtype=np.float32).astype(dtype)
    if kind == "lattice":
        return inputs.sc_lattice(round(n ** (1.0 / 3.0)), L=L, perturb=1e-3 * L / round(n ** (1.0 / 3.0)), seed=1,
                                 dtype=np.float32).astype(dtype)
    return inputs.clustered(n, L=L, seed=n, dtype=np.float32).astype(dtype)


@pytest.mark.parametrize("tpc", [0, 4, 8])
@pytest.mark.parametrize("kind,n,dtype,periodic", [
    ("uniform", 1, np.float32, False), ("uniform", 31, np.float32, False), ("uniform", 33, np.float64, False),
    ("uniform", 1000, np.float32, True), ("uniform", 4097, np.float64, True), ("clustered", 9001, np.float32, False),
    ("uniform", 65535, np.float32, True), ("uniform", 65536, np.float64, False), ("clustered", 70001, np.float32, True),
    ("clustered", 66001, np.float64, False), ("lattice", 42 ** 3, np.float32, True),
    ("uniform", 2097152 + 33, np.float32, True)])
def test_same_bits_as_the_warp_kernel(kind, n, dtype, periodic, tpc):
    L = float(np.float32(100.0 * (n / 2097152.0) ** (1.0 / 3.0))) if kind == "clustered" else 1.0
    pos = torch.from_numpy(points(kind, n, dtype, L)).cuda()
    box = ((0.0,) * 3, (L,) * 3)
    ref = outputs(vt.vt_build(pos, None, *box, periodic, threads_per_cell=32))
    h = vt.vt_build(pos, None, *box, periodic, threads_per_cell=tpc)
    same(outputs(h), ref)
    st = vt.vt_status(h)
    assert st["rc"] == 0 and st["n_faces"] == len(ref["ids"])
    # the same handle again, on other points and back
    vt.vt_rebuild(h, (L - pos).clamp(0.0, L * (1.0 - 1e-6)) if n > 1 else pos)
    vt.vt_rebuild(h, pos)
    same(outputs(h), ref)


def test_sets_that_share_buckets_with_mixed_modes():
    pts, off = inputs.halo_sets(n_sets=60, nmin=1, nmax=5000, seed=21)
    pos = torch.from_numpy(pts).cuda()
    n = len(off) - 1
    boxes = np.tile([-1.0, -1.0, -1.0, 1.0, 1.0, 1.0], (n, 1))
    ref = outputs(vt.vt_build_batched(pos, off, boxes, threads_per_cell=32))
    for tpc in (4, 8):
        same(outputs(vt.vt_build_batched(pos, off, boxes, threads_per_cell=tpc)), ref)
    g = np.random.default_rng(3)
    set_k = g.choice([16, 24, 48, 64], n).astype(np.int32)
    ref = outputs(vt.vt_build_batched(pos, off, boxes, set_k=set_k, set_tpc=np.full(n, 32, np.int32)))
    mixed = g.choice([4, 8, 32], n).astype(np.int32)
    same(outputs(vt.vt_build_batched(pos, off, boxes, set_k=set_k, set_tpc=mixed)), ref)


def test_owned_rows_above_the_threshold():
    x = inputs.uniform(70000, seed=5, dtype=np.float32)
    pos = torch.from_numpy(x).cuda()
    full = vt.vt_build(pos, None)
    part = vt.vt_build_owned(pos, 40001, None)
    v, r = vt.cells(full)[0], vt.cell_radius(full)
    pv, pr = vt.cells(part)[0], vt.cell_radius(part)
    assert torch.equal(pv[:40001], v[:40001]) and torch.equal(pr[:40001], r[:40001])
    assert not pv[40001:].any() and not pr[40001:].any()


def test_errors_come_back_from_the_handed_over_cells():
    x = inputs.uniform(65536, seed=6, dtype=np.float32)
    x[60000] = x[17]
    with pytest.raises(vt.VTError) as e:
        vt.vt_build(torch.from_numpy(x).cuda(), None)
    assert e.value.code == vt.VT_ERR_DUPLICATE
    c = inputs.clustered(65536, L=31.5, seed=1)
    with pytest.raises(vt.VTError) as e:
        vt.vt_build(torch.from_numpy(c).cuda(), None, (0.0,) * 3, (31.5,) * 3, True, max_passes=1)
    assert e.value.code == vt.VT_ERR_SECURITY


def test_without_room_for_lane_groups_a_warp_takes_each_cell():
    """The lane-group kernels' memory is allocated last; where it fails the library's own choice falls back."""
    pos = torch.from_numpy(inputs.uniform(65536, seed=9).astype(np.float64)).cuda()
    ref = outputs(vt.vt_build(pos, None))
    fell_back = 0
    for nth in range(1, 64):
        vt.vt_debug_fail_alloc(nth)
        try:
            h = vt.vt_build(pos, None)
        except vt.VTError as e:
            assert e.code == vt.VT_ERR_OOM and not fell_back
            continue
        if vt.vt_debug_fail_alloc(0):
            break
        fell_back += 1
        same(outputs(h), ref)
    assert fell_back == 7
    vt.vt_debug_fail_alloc(20)
    with pytest.raises(vt.VTError):
        vt.vt_build(pos, None)
    for nth in range(21, 32):  # an explicit choice does not fall back
        vt.vt_debug_fail_alloc(nth)
        try:
            vt.vt_build(pos, None, threads_per_cell=8)
            assert vt.vt_debug_fail_alloc(0) > 0
        except vt.VTError as e:
            assert e.code == vt.VT_ERR_OOM


def test_a_facet_pool_of_exactly_the_facets():
    """A perturbed BCC lattice has 14 facets per cell: a pool of 14 records per particle is just enough, and too small
    for uniform points (15.5 on average)."""
    lat = torch.from_numpy(inputs.bcc_lattice(32, perturb=1e-4, seed=2, dtype=np.float32)).cuda()
    h = vt.vt_build(lat, None, face_pool=14)
    vt.vt_rebuild(h, torch.from_numpy(inputs.uniform(len(lat), seed=4, dtype=np.float32)).cuda())
    assert vt.vt_status(h)["rc"] == vt.VT_ERR_CAPACITY
    vt.vt_rebuild(h, lat)
    assert vt.vt_status(h)["rc"] == 0
