"""Lane groups that the library chose by itself give their memory (up to 5.4 GB) back where a later allocation of the
handle fails: the facet pool that has to grow during a build, or what a product asks for at its first call.  A warp then takes
each cell, with the same bits.  Failures are injected on the host (vt_debug_fail_alloc).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1601_06429_gb300 import binding as vt
from paper_1601_06429_gb300 import inputs

pytestmark = pytest.mark.gpu
N = 65536


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1601_06429_gb300.build import build

    build()
    vt.load_library()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.fixture(autouse=True)
def _disarm():
    yield
    vt.vt_debug_fail_alloc(0)


def same(a, b):
    return all(torch.equal(p, q) for p, q in zip(vt.cells(a), vt.cells(b))) and torch.equal(vt.gradient(a), vt.gradient(b))


def test_the_facet_pool_grows_in_place_of_lane_groups():
    pos = torch.from_numpy(inputs.uniform(N, seed=3, dtype=np.float32)).cuda()
    ref = vt.vt_build(pos, None)
    fired = 0
    for nth in range(1, 64):
        vt.vt_debug_fail_alloc(nth)
        try:
            h = vt.vt_build(pos, None, face_pool=1)
        except vt.VTError as e:
            assert e.code == vt.VT_ERR_OOM and not fired  # the workspace itself, before any of this memory
            continue
        if vt.vt_debug_fail_alloc(0):
            break
        fired += 1
        assert same(h, ref)
        vt.vt_rebuild(h, pos)
        assert same(h, ref) and vt.vt_status(h)["rc"] == 0
    assert fired == 7  # the six arrays of the lane groups, and the larger pool
    vt.vt_debug_fail_alloc(nth - 1)  # lane groups asked for by name stay
    with pytest.raises(vt.VTError) as e:
        vt.vt_build(pos, None, face_pool=1, threads_per_cell=4)
    assert e.value.code == vt.VT_ERR_OOM


def test_products_take_the_room_of_lane_groups():
    pos = torch.from_numpy(inputs.uniform(N, seed=4, dtype=np.float32)).cuda()
    ref = vt.vt_build(pos, None)
    grid = vt.grid_density_volume(ref, 16)
    h = vt.vt_build(pos, None)
    vt.vt_debug_fail_alloc(1)
    got = vt.grid_density_volume(h, 16)
    assert vt.vt_debug_fail_alloc(0) == 0
    assert (got - grid).abs().max() <= 1e-6 * grid.abs().max()
    other = torch.from_numpy(inputs.uniform(N, seed=5, dtype=np.float32)).cuda()
    vt.vt_rebuild(h, other)
    vt.vt_rebuild(h, pos)
    assert same(h, ref)


def test_a_captured_rebuild_keeps_its_memory():
    pos = torch.from_numpy(inputs.uniform(N, seed=6, dtype=np.float32)).cuda()
    ref = vt.vt_build(pos, None)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        h = vt.vt_build(pos, None, stream=s)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        vt.vt_rebuild(h, pos)
    vt.vt_debug_fail_alloc(1)
    with pytest.raises(vt.VTError) as e:
        vt.grid_density_volume(h, 16)
    assert e.value.code == vt.VT_ERR_OOM
    g.replay()
    torch.cuda.synchronize()
    assert vt.vt_status(h)["rc"] == 0 and same(h, ref)


@pytest.mark.parametrize("tpc,set_tpc,falls_back", [
    (4, 0, True), (4, None, False), (0, None, True), (0, 4, False), (32, (1, 0), True), (0, (1, 8), False)])
def test_whose_choice_lane_groups_of_a_batch_are(tpc, set_tpc, falls_back):
    """The last allocation of a batch that takes lane groups is theirs: set_tpc (0: the library's choice), where it is
    given, replaces threads_per_cell."""
    n = 2
    off = np.array([0, N // 2, N + 1000], np.int64)
    pos = torch.from_numpy(inputs.uniform(int(off[-1]), seed=7, dtype=np.float32)).cuda()
    boxes = np.tile([0.0, 0.0, 0.0, 1.0, 1.0, 1.0], (n, 1))
    kw = {"threads_per_cell": tpc}
    if set_tpc is not None:
        kw["set_tpc"] = np.broadcast_to(np.array(set_tpc, np.int32), (n,)).copy()
    vol = vt.cells(vt.vt_build_batched(pos, off, boxes, **kw))[0]
    vt.vt_debug_fail_alloc(1000)
    vt.vt_destroy(vt.vt_build_batched(pos, off, boxes, **kw))
    last = 1000 - vt.vt_debug_fail_alloc(0)
    vt.vt_debug_fail_alloc(last)
    if falls_back:
        h = vt.vt_build_batched(pos, off, boxes, **kw)
        assert vt.vt_debug_fail_alloc(0) == 0
        assert torch.equal(vt.cells(h)[0], vol)
    else:
        with pytest.raises(vt.VTError) as e:
            vt.vt_build_batched(pos, off, boxes, **kw)
        assert e.value.code == vt.VT_ERR_OOM
