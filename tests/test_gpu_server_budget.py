"""Admission under a tight memory budget: a volume fits without the tile records
that only speed its queries up, and answers the same."""
import numpy as np
import pytest

import oracle
from paper_2009_02702_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS, S = (128, 96, 80), 40


@pytest.fixture(scope="module")
def mg():
    from paper_2009_02702_gb300 import mg as _mg
    _mg.lib()
    return _mg


def admitted(mg, g, hist, budget):
    srv = mg.Server(slots=2, max_batch=64, hist=hist, memory_budget=budget)
    try:
        srv.add_volume(g, 4)
    except mg.MGError as e:
        assert e.status == mg.MG_ERR_CAPACITY
        srv.close()
        return None
    assert budget == 0 or srv.stats()["memory_admitted"] <= budget
    return srv


@pytest.mark.parametrize("hist", ["u32", "f32"])
def test_volume_admitted_without_its_tiles(mg, hist):
    vol = synth.make_volume(2, dims=DIMS, S=S)
    ids = torch.from_numpy(vol).cuda()
    g = mg.mg_build(ids, S)
    srv = admitted(mg, g, hist, 0)
    full = srv.stats()["memory_admitted"]
    srv.close()
    with_tiles = mg.mg_graph_info_get(g)["device_bytes"]
    # the graph's tiles are in use now: it is admitted with shorter maps or not at all
    srv = admitted(mg, g, hist, full)
    assert srv is not None
    srv.close()
    fresh = mg.mg_build(ids, S)
    lo = with_tiles // 2
    hi = full
    while hi - lo > 1024:   # the least budget that a fresh graph is admitted with
        mid = (lo + hi) // 2
        h = mg.mg_build(ids, S)
        srv = admitted(mg, h, hist, mid)
        lo, hi = (lo, mid) if srv else (mid, hi)
        if srv:
            srv.close()
        h.close()
    srv = admitted(mg, fresh, hist, hi)
    bare = mg.mg_graph_info_get(fresh)["device_bytes"]
    voxels = DIMS[0] * DIMS[1] * DIMS[2]
    assert bare < with_tiles - voxels // 2          # the records are gone: at least half a byte a voxel
    assert admitted(mg, g, hist, hi) is None        # ... but never from under a graph that has been queried
    boxes = synth.make_boxes(1, 50, dims=DIMS, box_max=128)
    ref = oracle.box_hist(vol, S, boxes)
    tickets = [srv.submit_box(0, b) for b in boxes]
    srv.start()
    for k, (t, out) in enumerate(tickets):
        srv.wait(t, timeout=30.0)
        assert np.array_equal(out.astype(np.int64), ref[k].astype(np.int64)), k
    srv.close()
    t = torch.from_numpy(boxes).cuda()
    for alpha in ("f32", "f16"):
        h = mg.mg_query_boxes(fresh, t, hist="f32", alpha=alpha).cpu().numpy().astype(np.float64)
        tol = 0.0 if alpha == "f32" else 1.5 * fresh.info["depth"] * 2.0 ** -11
        assert (np.abs(h - ref).sum(1) <= tol * ref.sum(1)).all()
    mg.mg_sync_status(fresh)
    g.close()
    fresh.close()
